// FP64 Grams and block products on the tensor cores.
//
// GB300's FP64 pipe is 1/64 of its FP32 rate, and the FP64 contractions of the
// all-FP64 mode, the orthonormalization and the Rayleigh-Ritz step ran at that
// pipe's peak. Here an FP64 column is cut into eight 8-bit digits against the
// largest exponent of the column (the error-free slicing of Ozaki, Ogita,
// Oishi and Rump, "Error-free transformations of matrix multiplication by
// using fast routines of matrix multiplication and its applications",
// Numerical Algorithms 59, 2012, in the integer form for low-precision matrix
// units): x = 2^(e - 62) q + r with |r| <= 2^(e - 63) and
// q = sum_d s_d 2^(8 (7 - d)), |s_d| <= 128. The digits are exact in BF16 and a
// product of two is at most 2^14, so the FP32 accumulator of the BF16 MMA holds
// every sum of up to kChunk * 32 rows of all products of equal weight exactly
// (8 * 128 * 2^14 = 2^24): nothing is rounded until the integer sums, held in
// 64 bits, are turned into one FP64 value. Dropped are r and the products of
// weight below 2^-56 of the leading one (36 of 64 are kept): per term of a sum
// less than 2^-57 max|a| max|b| of the two columns, usually about 2^-61. That is
// FP64 norm-wise, for any block: a sum of random terms, or of columns whose
// largest entry is up to 2^8 times their usual one, is no further off than an
// FP64 chain leaves it (measured: at most as far for every FP64 call of the
// repository's sizes; seven-bit digits, 2^-55, were 2.3 times further off at max
// / rms = 8). It is not FP64 entry by entry: entries below 2^-9 of their column's
// largest lose low bits and those below 2^-63 of it vanish, so in a column that
// falls off exponentially the small entries of a product carry an error
// relative to the large ones.
//
// One CTA owns a 128 x 64 output tile: eight accumulators (one per weight) of
// 64 columns fill the 512 TMEM columns. Per 32-deep stage TMA brings all eight
// digits of the A (64 KB) and B (32 KB) tiles, two stages in flight, and one
// thread issues the 72 MMAs. What bounds the kernel is the shared memory that
// a 128 x 64 MMA reads (6 KB per 131072 multiply-adds).
//
// Warp roles (576 threads): warp 0 TMA, warp 1 TMEM allocation and MMA, warps
// 2-17 take a finished chunk out of TMEM into 64-bit sums (four warps per lane
// quarter, 16 columns each) and write the result. Every mbarrier wait is
// bounded (bit 2 of *err), as in the other tensor-core kernels.
#include <cooperative_groups.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <atomic>

#include "ops.cuh"
#include "tc.cuh"

namespace trm {

namespace {

using namespace tc;
namespace cg = cooperative_groups;

constexpr int ND = 8;          // digits
constexpr int OM = 128;        // tile rows (MMA M)
constexpr int ON = 64;         // tile columns (MMA N)
constexpr int OK = 32;         // contraction depth of a stage
constexpr int kChunk = 4;      // stages an accumulator may sum exactly
constexpr int OSTAGES = 2;
constexpr int EPIW = 16;        // warps that read the accumulators
constexpr int EC = ON * 4 / EPIW;  // columns of each
constexpr int OTHREADS = 64 + 32 * EPIW;
constexpr int ABYTES = ND * OM * OK * 2, BBYTES = ND * ON * OK * 2;

struct OzSmem {
  unsigned char a[OSTAGES][ABYTES];  // [digit][128 columns][32 rows], or
                                     // [row half][digit][32 columns][64 rows]
  unsigned char b[OSTAGES][BBYTES];  // [digit][64 columns][32 rows]
  uint64_t full[OSTAGES], empty[OSTAGES], accfull, accempty, mmadone;
  uint32_t tmem_base;
  int failed;
  double red[4 * 32];
};

// ---------------------------------------------------------------------------
// Digits of a block's columns
// ---------------------------------------------------------------------------
// q of x against the exponent field E of the column's largest magnitude:
// x 2^(62 - e) rounded, e = E - 1022.
__device__ __forceinline__ long long oz_fixed(double x, int E) {
  const long long u = __double_as_longlong(x);
  const int ex = (int)((u >> 52) & 0x7FF);
  if (ex == 0) return 0;  // zero (or below 2^-1022 of anything in the sum)
  const long long mant = (u & 0xFFFFFFFFFFFFFll) | (1ll << 52);
  const int sh = E - ex - 9;
  long long q;
  if (sh <= 0)
    q = mant << -sh;  // sh >= -9
  else if (sh < 54)
    q = (mant + (1ll << (sh - 1))) >> sh;
  else
    q = 0;
  return u < 0 ? -q : q;
}
// Digit d of q as BF16 bits; u = q plus 128 in each of the lower seven digits.
// The float conversion is exact: 2^23 + 128 + digit, minus 2^23 + 128.
__device__ __forceinline__ uint32_t oz_digit(unsigned long long u, int d) {
  float f;
  if (d == 0)
    f = (float)(int)((long long)u >> 56);
  else
    f = __uint_as_float(0x4B000000u | ((uint32_t)(u >> (8 * (7 - d))) & 255u)) -
        8388736.0f;
  return __float_as_uint(f) >> 16;
}
constexpr unsigned long long kDigitBias = 0x0080808080808080ull;

// Source of a sliced column: C, or fc C + fp P (columns ld apart), with fp =
// sc->alpha when sc is given.
struct OzSrc {
  const double* c;
  const double* p;
  const IterScalars* sc;
  double fc, fp;
  int64_t ld;
};

// Digits of column blockIdx.y, its rows shared by the cluster's CTAs: the
// largest exponent over the cluster, then 8 digits of four rows per thread and
// step. lds (a multiple of 8) rows are written, those past N as zeros.
// scale[j] = 2^(e - 16); NaN when the column holds an infinity or NaN.
__global__ void __launch_bounds__(512)
    k_oz_slice(int64_t N, int64_t lds, int64_t sstride, OzSrc src,
               __nv_bfloat16* __restrict__ out, double* __restrict__ scale) {
  __shared__ int mx;
  const cg::cluster_group cl = cg::this_cluster();
  const int parts = gridDim.x, part = blockIdx.x, j = blockIdx.y;
  const int64_t quads = lds >> 2, per = (quads + parts - 1) / parts;
  const int64_t q0 = part * per, q1 = min(quads, q0 + per);
  const double* c = src.c + (int64_t)j * src.ld;
  const double* p = src.p ? src.p + (int64_t)j * src.ld : nullptr;
  const double fp = src.sc ? src.sc->alpha : src.fp, fc = src.fc;
  const bool vec = ((reinterpret_cast<uintptr_t>(c) |
                     reinterpret_cast<uintptr_t>(p)) & 15) == 0;
  auto load = [&](int64_t q, double (&v)[4]) {
    const int64_t i = 4 * q;
    if (vec && i + 3 < N) {
      const double2 a = *reinterpret_cast<const double2*>(c + i);
      const double2 b = *reinterpret_cast<const double2*>(c + i + 2);
      v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
      if (p) {
        const double2 e = *reinterpret_cast<const double2*>(p + i);
        const double2 f = *reinterpret_cast<const double2*>(p + i + 2);
        v[0] = fma(fp, e.x, fc * v[0]); v[1] = fma(fp, e.y, fc * v[1]);
        v[2] = fma(fp, f.x, fc * v[2]); v[3] = fma(fp, f.y, fc * v[3]);
      }
    } else {
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        v[k] = i + k < N ? c[i + k] : 0.0;
        if (p && i + k < N) v[k] = fma(fp, p[i + k], fc * v[k]);
      }
    }
  };
  if (threadIdx.x == 0) mx = 0;
  __syncthreads();
  int m = 0;
#pragma unroll 2
  for (int64_t q = q0 + threadIdx.x; q < q1; q += blockDim.x) {
    double v[4];
    load(q, v);
#pragma unroll
    for (int k = 0; k < 4; ++k)
      m = max(m, (int)(__double2hiint(v[k]) & 0x7FFFFFFF));
  }
  m = __reduce_max_sync(0xffffffffu, m);
  if ((threadIdx.x & 31) == 0) atomicMax(&mx, m);
  cl.sync();
  int E = 0;
  for (int r = 0; r < parts; ++r) E = max(E, *cl.map_shared_rank(&mx, r));
  cl.sync();  // no CTA leaves while another reads its maximum
  E >>= 20;   // the exponent field
  if (part == 0 && threadIdx.x == 0)
    scale[j] = E == 2047 ? __longlong_as_double(0x7FF8000000000000ll)
               : E == 0  ? 0.0
                         : ldexp(1.0, E - 1022 - 16);
  const bool zero = E == 0 || E == 2047;
#pragma unroll 2
  for (int64_t q = q0 + threadIdx.x; q < q1; q += blockDim.x) {
    double v[4];
    load(q, v);
    unsigned long long u[4];
#pragma unroll
    for (int k = 0; k < 4; ++k)
      u[k] = (unsigned long long)(zero ? 0ll : oz_fixed(v[k], E)) + kDigitBias;
    __nv_bfloat16* o = out + (int64_t)j * lds + 4 * q;
#pragma unroll
    for (int d = 0; d < ND; ++d) {
      uint2 w;
      w.x = oz_digit(u[0], d) | (oz_digit(u[1], d) << 16);
      w.y = oz_digit(u[2], d) | (oz_digit(u[3], d) << 16);
      *reinterpret_cast<uint2*>(o + d * sstride) = w;
    }
  }
}

// Digits of the small factor of a product, M' = diag(2^16 scale) M (k x n FP64,
// ld k): column j on CTA j, out[d][j][ldk], zeros past k. fscale as scale.
__global__ void __launch_bounds__(128)
    k_oz_slice_small(int k, int ldk, const double* __restrict__ M,
                     const double* __restrict__ scale,
                     __nv_bfloat16* __restrict__ out, double* __restrict__ fscale) {
  __shared__ int mx;
  const int j = blockIdx.x, n = gridDim.x;
  if (threadIdx.x == 0) mx = 0;
  __syncthreads();
  const double* c = M + (size_t)j * k;
  int m = 0;
  for (int i = threadIdx.x; i < k; i += blockDim.x)
    m = max(m, (int)(__double2hiint(c[i] * (scale[i] * 65536.0)) & 0x7FFFFFFF));
  m = __reduce_max_sync(0xffffffffu, m);
  if ((threadIdx.x & 31) == 0) atomicMax(&mx, m);
  __syncthreads();
  const int E = mx >> 20;
  if (threadIdx.x == 0)
    fscale[j] = E == 2047 ? __longlong_as_double(0x7FF8000000000000ll)
                : E == 0  ? 0.0
                          : ldexp(1.0, E - 1022 - 16);
  const bool zero = E == 0 || E == 2047;
  for (int i = threadIdx.x; i < ldk; i += blockDim.x) {
    const double v = i < k ? c[i] * (scale[i] * 65536.0) : 0.0;
    const unsigned long long u =
        (unsigned long long)(zero ? 0ll : oz_fixed(v, E)) + kDigitBias;
#pragma unroll
    for (int d = 0; d < ND; ++d) {
      const uint16_t w = (uint16_t)oz_digit(u, d);
      reinterpret_cast<uint16_t*>(out)[((size_t)d * n + j) * ldk + i] = w;
    }
  }
}

// ---------------------------------------------------------------------------
// The contraction
// ---------------------------------------------------------------------------
enum OzMode { kOzGram = 0, kOzStore = 1, kOzGrad = 2 };

struct OzArgs {
  // Gram: rows of this launch's slices; product: N rows in 128-row tiles
  int64_t N;
  int m, n;                // Gram: out m x n per segment; product: k = m, n
  int64_t rows_per_split;  // Gram
  int tiles_m, tiles_n;    // Gram: per segment; product: row tiles, column tiles
  int tri;                 // product: the small factor is upper triangular
  const double* sa[2];     // Gram: column scales of A (per segment) and B
  const double* sb;        // product: scales of the small factor's columns
  double* part;            // Gram partials; gradient: four sums per CTA
  double* out;             // product, columns ldo apart
  int64_t ldo;
  const double* xp;        // gradient
  const double* gprev;
  const double* pprev;
  const double* minv;
  int* err;
  const int* halt;         // product (may be null): nothing is written when
                           // bit 1 of *halt is set
};

// BF16 instruction descriptor, FP32 accumulation; a_mn: A is MN-major.
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N, bool a_mn) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((a_mn ? 1u : 0u) << 15) |
         ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}
__device__ __forceinline__ void mma_bf16(uint32_t d, uint64_t a, uint64_t b,
                                         uint32_t idesc, uint32_t accum) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d),
      "l"(a), "l"(b), "r"(idesc), "r"(accum));
}
__device__ __forceinline__ void tma_load_3d(void* dst, const CUtensorMap* map,
                                            int x, int y, int z,
                                            uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::"
      "complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z),
      "r"(smem_u32(bar))
      : "memory");
}
// K-major operand: lines of 32 values (64 bytes, 64-byte swizzle), groups of
// eight lines 512 bytes apart.
__device__ __forceinline__ uint64_t oz_kdesc(uint32_t saddr) {
  return (uint64_t)((saddr & 0x3FFFF) >> 4) | ((uint64_t)1 << 16) |
         ((uint64_t)(512 >> 4) << 32) | ((uint64_t)1 << 46) |
         ((uint64_t)4 << 61);
}
// MN-major operand: lines of 64 rows (128 bytes, 128-byte swizzle), eight
// lines along K 1024 bytes apart, the second 64 rows `half` bytes on.
__device__ __forceinline__ uint64_t oz_mndesc(uint32_t saddr, uint32_t half) {
  return smem_desc(saddr, half, 1024);
}

template <int MODE>
__global__ void __launch_bounds__(OTHREADS, 1)
    k_oz(const __grid_constant__ CUtensorMap mapA0,
         const __grid_constant__ CUtensorMap mapA1,
         const __grid_constant__ CUtensorMap mapB, OzArgs args) {
  extern __shared__ unsigned char smem_raw[];
  OzSmem* sm = reinterpret_cast<OzSmem*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  constexpr bool gram = MODE == kOzGram;
  if (MODE == kOzStore && args.halt && (*args.halt & 1)) return;
  // Jobs: Gram, one (split, tile); products, tiles blockIdx.x, + gridDim.x, ...
  // with the column tile fastest (the tiles of a row tile share A in L2).
  const int njobs = gram ? 1 : args.tiles_m * args.tiles_n;
  const int first = gram ? 0 : blockIdx.x, step = gram ? 1 : gridDim.x;
  struct Job {
    int i0, j0, seg, nst;  // tile origin, A segment, stages
    int64_t rb;            // Gram: first row
  };
  auto job = [&](int t) {
    Job g;
    if (gram) {
      const int tile = blockIdx.y, per = args.tiles_m * args.tiles_n;
      g.seg = tile / per;
      const int r = tile - g.seg * per;
      g.i0 = (r % args.tiles_m) * OM;
      g.j0 = (r / args.tiles_m) * ON;
      g.rb = (int64_t)blockIdx.x * args.rows_per_split;
      const int64_t re = min(args.N, g.rb + args.rows_per_split);
      g.nst = (int)((re - g.rb + OK - 1) / OK);
    } else {
      g.seg = 0;
      // (a grid that is a multiple of the column tiles would give a CTA the
      // same one every time, and an upper triangular factor's differ in work)
      const int turn = gridDim.x % args.tiles_n == 0 ? t / gridDim.x : 0;
      g.i0 = (t / args.tiles_n) * OM;
      g.j0 = ((t + turn) % args.tiles_n) * ON;
      g.rb = 0;
      // an upper triangular factor: column j needs the rows k <= j
      const int k = args.tri ? min(args.m, g.j0 + ON) : args.m;
      g.nst = (k + OK - 1) / OK;
    }
    return g;
  };

  if (threadIdx.x == 0) {
    for (int s = 0; s < OSTAGES; ++s) {
      mbar_init(&sm->full[s], 1);
      mbar_init(&sm->empty[s], 1);
    }
    mbar_init(&sm->accfull, 1);
    mbar_init(&sm->accempty, 32 * EPIW);
    mbar_init(&sm->mmadone, 1);
    sm->failed = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) tmem_alloc(&sm->tmem_base, 512);
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = sm->tmem_base;

  if (warp == 0) {
    if (lane == 0) {
      int it = 0;
      bool ok = true;
      for (int t = first; t < njobs && ok; t += step) {
        const Job g = job(t);
        const CUtensorMap* ma = g.seg ? &mapA1 : &mapA0;
        for (int k = 0; k < g.nst; ++k, ++it) {
          const int s = it % OSTAGES;
          if (it >= OSTAGES && !mbar_wait(&sm->empty[s], ((it / OSTAGES) - 1) & 1,
                                          args.err, &sm->failed)) {
            ok = false;
            break;
          }
          mbar_expect_tx(&sm->full[s], ABYTES + BBYTES);
          if (gram) {
            const int x = (int)(g.rb + (int64_t)k * OK);
            tma_load_3d(sm->a[s], ma, x, g.i0, 0, &sm->full[s]);
            tma_load_3d(sm->b[s], &mapB, x, g.j0, 0, &sm->full[s]);
          } else {
            tma_load_3d(sm->a[s], ma, g.i0, k * OK, 0, &sm->full[s]);
            tma_load_3d(sm->a[s] + ABYTES / 2, ma, g.i0 + 64, k * OK, 0,
                        &sm->full[s]);
            tma_load_3d(sm->b[s], &mapB, k * OK, g.j0, 0, &sm->full[s]);
          }
        }
      }
      // the copies in flight must land before the CTA may exit
      for (int j = it > OSTAGES ? it - OSTAGES : 0; j < it; ++j)
        mbar_wait_own(&sm->full[j % OSTAGES], (j / OSTAGES) & 1, args.err);
    }
  } else if (warp == 1) {
    if (lane == 0) {
      constexpr uint32_t idesc = idesc_bf16(OM, ON, !gram);
      int it = 0, ch = 0;
      bool ok = true;
      for (int t = first; t < njobs && ok; t += step) {
        const Job g = job(t);
        for (int k = 0; k < g.nst && ok; ++k, ++it) {
          const int s = it % OSTAGES, kc = k % kChunk;
          if (kc == 0 && ch > 0 && !mbar_wait(&sm->accempty, (ch - 1) & 1,
                                              args.err, &sm->failed)) {
            ok = false;
            break;
          }
          if (!mbar_wait(&sm->full[s], (it / OSTAGES) & 1, args.err,
                         &sm->failed)) {
            ok = false;
            break;
          }
          fence_after();
          // (digit pairs by A digit: neighbouring MMAs go to different
          // accumulators; the descriptors differ by constants in their
          // address field, so an MMA costs the issuing thread few instructions)
          const uint64_t a0 = gram ? oz_kdesc(smem_u32(sm->a[s]))
                                   : oz_mndesc(smem_u32(sm->a[s]), ABYTES / 2);
          const uint64_t b0 = oz_kdesc(smem_u32(sm->b[s]));
          const uint32_t more = kc > 0 ? 1u : 0u;
#pragma unroll
          for (int i = 0; i < ND; ++i)
#pragma unroll
            for (int j = 0; j < ND - i; ++j)
#pragma unroll
              for (int kk = 0; kk < OK / 16; ++kk)
                mma_bf16(tmem + (uint32_t)((i + j) * ON),
                         a0 + (gram ? (i * (OM * 64) + kk * 32) >> 4
                                    : (i * 4096 + kk * 2048) >> 4),
                         b0 + ((j * (ON * 64) + kk * 32) >> 4), idesc,
                         (i > 0 || kk > 0) ? 1u : more);
          mma_commit(&sm->empty[s]);
          if (kc == kChunk - 1 || k == g.nst - 1) {
            mma_commit(&sm->accfull);
            ++ch;
          }
        }
      }
      mma_commit(&sm->mmadone);
      mbar_wait_own(&sm->mmadone, 0, args.err);
    }
  } else {
    const int q = warp & 3;                 // TMEM lane quarter
    const int c0 = EC * ((warp - 2) >> 2);  // first of its columns
    const int rr = 32 * q + lane;
    const uint32_t lrow = (uint32_t)(32 * q) << 16;
    double s_gg = 0.0, s_gmg = 0.0, s_pmg = 0.0, s_gpp = 0.0;
    int ch = 0;
    bool ok = true;
    for (int t = first; t < njobs && ok; t += step) {
      const Job g = job(t);
      const int nch = (g.nst + kChunk - 1) / kChunk;
      // T1 = sum_{d<4} v_d 2^(8 (3 - d)), T2 = sum_{d>=4} v_d 2^(8 (7 - d))
      long long t1[EC], t2[EC];
#pragma unroll
      for (int e = 0; e < EC; ++e) t1[e] = t2[e] = 0;
      for (int c = 0; c < nch; ++c, ++ch) {
        const bool got = mbar_wait(&sm->accfull, ch & 1, args.err, &sm->failed);
        if (!__all_sync(0xffffffffu, got)) {  // TMEM loads are .sync.aligned
          ok = false;
          break;
        }
        fence_after();
#pragma unroll
        for (int d = 0; d < ND; ++d) {
          uint32_t x[EC];
          tmem_ld16(tmem + lrow + (uint32_t)(d * ON + c0), x);
#pragma unroll
          for (int e = 0; e < EC; ++e) {
            const int v = __float2int_rn(__uint_as_float(x[e]));
            if (d < 4)
              t1[e] += (long long)v * (1 << (8 * (3 - d)));
            else
              t2[e] += (long long)v * (1 << (8 * (7 - d)));
          }
        }
        fence_before();
        mbar_arrive(&sm->accempty);
      }
      if (!ok) break;
      const int row = g.i0 + rr;
      if (gram) {
        double* out = args.part +
                      ((size_t)blockIdx.x * (gridDim.y / (args.tiles_m * args.tiles_n)) +
                       g.seg) * args.m * args.n;
        const double sa = row < args.m ? args.sa[g.seg][row] : 0.0;
#pragma unroll
        for (int e = 0; e < EC; ++e) {
          const int col = g.j0 + c0 + e;
          if (row < args.m && col < args.n) {
            // (T1 + 2^-32 T2) 2^(ea + eb - 36)
            const double v =
                fma((double)t2[e], 0x1p-36, 0x1p-4 * (double)t1[e]);
            out[row + (size_t)col * args.m] = v * sa * args.sb[col];
          }
        }
      } else {
        const double mi = MODE == kOzGrad && args.minv && row < args.N
                              ? args.minv[row] : 1.0;
#pragma unroll 4
        for (int e = 0; e < EC; ++e) {
          const int col = g.j0 + c0 + e;
          if (row < args.N && col < args.n) {
            // the integers are below 2^51: exact through the 2^52 bias
            const double h1 = __longlong_as_double(0x4338000000000000ll + t1[e]) -
                              __longlong_as_double(0x4338000000000000ll);
            const double h2 = __longlong_as_double(0x4338000000000000ll + t2[e]) -
                              __longlong_as_double(0x4338000000000000ll);
            const double v = fma(h2, 0x1p-32, h1);
            const double f = args.sb[col] * 0x1p-20;  // 2^(f_j - 36)
            const int64_t o = row + (int64_t)col * args.ldo;
            if (MODE == kOzStore) {
              args.out[o] = v * f;
            } else {
              const double gg = fma(2.0 * f, v, -2.0 * args.xp[o]);
              args.out[o] = gg;
              const double mg = mi * gg;
              s_gg = fma(gg, gg, s_gg);
              s_gmg = fma(gg, mg, s_gmg);
              if (args.gprev) s_pmg = fma(args.gprev[o], mg, s_pmg);
              if (args.pprev) s_gpp = fma(gg, args.pprev[o], s_gpp);
            }
          }
        }
      }
    }
    __syncwarp();
    if (MODE == kOzGrad) {  // the CTA's four sums, in a fixed order
      double v[4] = {s_gg, s_gmg, s_pmg, s_gpp};
      const double w = warp_sum4(v);
      if ((lane & 7) == 0) sm->red[(lane >> 3) * 32 + warp - 2] = w;
      asm volatile("bar.sync 1, %0;" ::"n"(32 * EPIW) : "memory");
      if (warp < 6) {
        const double x = warp_sum(lane < EPIW ? sm->red[(warp - 2) * 32 + lane] : 0.0);
        if (lane == 0) args.part[(size_t)blockIdx.x * 4 + warp - 2] = x;
      }
    }
  }
  __syncwarp();
  fence_before();
  __syncthreads();
  if (warp == 1) {
    __syncwarp();
    fence_after();
    tmem_dealloc(tmem, 512);
  }
}

// Digit array [digit][column][row] as a 3-D tensor map.
CUtensorMap oz_map(const __nv_bfloat16* p, int64_t rows, int cols, int64_t ld,
                   int64_t sstride, int box_rows, int box_cols, bool sw128) {
  EncodeFn fn = encode_fn();
  if (!fn) throw Error(-5, "cuTensorMapEncodeTiled is not available");
  CUtensorMap map;
  const cuuint64_t dims[3] = {(cuuint64_t)rows, (cuuint64_t)cols, ND};
  const cuuint64_t strides[2] = {(cuuint64_t)ld * 2, (cuuint64_t)sstride * 2};
  const cuuint32_t box[3] = {(cuuint32_t)box_rows, (cuuint32_t)box_cols, ND};
  const cuuint32_t estr[3] = {1, 1, 1};
  const CUresult r =
      fn(&map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3,
         const_cast<__nv_bfloat16*>(p), dims, strides, box, estr,
         CU_TENSOR_MAP_INTERLEAVE_NONE,
         sw128 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B,
         CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS)
    throw Error(-5, "cuTensorMapEncodeTiled failed: " + std::to_string((int)r));
  return map;
}

template <int MODE>
void oz_launch(dim3 grid, const CUtensorMap& a0, const CUtensorMap& a1,
               const CUtensorMap& b, const OzArgs& args, cudaStream_t s) {
  const size_t smem = sizeof(OzSmem) + 1024;
  static std::atomic<int> attr_dev{-1};  // launches may come from several threads
  int dev = 0;
  TRM_CUDA(cudaGetDevice(&dev));
  if (attr_dev.load(std::memory_order_relaxed) != dev) {
    TRM_CUDA(cudaFuncSetAttribute(k_oz<MODE>,
                                  cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)smem));
    attr_dev.store(dev, std::memory_order_relaxed);
  }
  k_oz<MODE><<<grid, OTHREADS, smem, s>>>(a0, a1, b, args);
  TRM_CHECK_LAUNCH();
}

int64_t oz_ld(int64_t N) { return (N + 7) & ~(int64_t)7; }
int oz_ldk(int k) { return (k + 7) & ~7; }

}  // namespace

// The slicing passes and whole 128 x 64 tiles cost about 50 us however small
// the product, the time of 3e7 multiply-adds on the FP64 pipe (110592 x 128:
// Gram 165 us and 98 for the digits of a block, against 3020; 32768 x 64: 51
// and 27, against 267).
bool oz_pays(int64_t N, int m, int n) {
  return (double)N * m * n >= 3e7 && N >= 1024 && m >= 8 && n >= 8 &&
         N < ((int64_t)1 << 31) - 128 && encode_fn() != nullptr;
}

size_t oz_block_bytes(int64_t N, int m) {
  return (size_t)ND * 2 * oz_ld(N) * m + 256;
}
size_t oz_small_bytes(int k, int n) {
  return (size_t)ND * 2 * oz_ldk(k) * n + 256;
}

void oz_slice(int64_t N, int m, const double* C, int64_t ldc, OzBlock& out,
              cudaStream_t s, const double* P, const IterScalars* sc, double fc,
              double fp) {
  out.N = N;
  out.m = m;
  const int64_t lds = oz_ld(N);
  // CTAs per column: about two waves of SMs, at most the portable cluster
  // size, at least a few thousand rows each
  int parts = 1;
  while (parts < 8 && (int64_t)parts * m < 2 * sm_count() &&
         N / (2 * parts) >= 2048)
    parts *= 2;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(parts, m);
  cfg.blockDim = dim3(512);
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = parts;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  TRM_CUDA(cudaLaunchKernelEx(&cfg, k_oz_slice, N, lds, lds * m,
                              OzSrc{C, P, sc, fc, fp, ldc},
                              static_cast<__nv_bfloat16*>(out.digits),
                              out.scale));
  TRM_CHECK_LAUNCH();
}

void oz_gram(const OzBlock* a, int segs, const OzBlock& b, double* out,
             double* partials, size_t cap, int* err, cudaStream_t s) {
  const int64_t N = b.N, lds = oz_ld(N);
  const int m = a[0].m, n = b.m;
  OzArgs g{};
  g.N = N;
  g.m = m;
  g.n = n;
  g.tiles_m = ceil_div(m, OM);
  g.tiles_n = ceil_div(n, ON);
  const int tiles = segs * g.tiles_m * g.tiles_n;
  const size_t count = (size_t)segs * m * n;
  // row slices: one wave of CTAs (each holds a whole SM), whole stages, as far
  // as the partials buffer goes; longer waves only where the tiles alone are one
  int64_t splits = std::max(1, sm_count() / tiles);
  splits = std::min<int64_t>(splits, ceil_div(N, (int64_t)4 * OK));
  // (the 64-bit sums hold 2^13 chunks of the largest digits)
  splits = std::max<int64_t>(splits, ceil_div(N, (int64_t)1 << 20));
  splits = std::min<int64_t>(splits, (int64_t)(cap / count));
  if (splits < 1 || ceil_div(N, splits) > (1 << 22)) throw Error(-2, "oz_gram: partials buffer too small");
  int64_t rows = ceil_div(N, splits);
  rows = ceil_div(rows, (int64_t)OK) * (int64_t)OK;
  splits = ceil_div(N, rows);
  g.rows_per_split = rows;
  g.sa[0] = a[0].scale;
  g.sa[1] = segs > 1 ? a[1].scale : nullptr;
  g.sb = b.scale;
  g.part = partials;
  g.err = err;
  auto map = [&](const OzBlock& x, int cols) {
    return oz_map(static_cast<const __nv_bfloat16*>(x.digits), lds, x.m, lds,
                  lds * x.m, OK, cols, false);
  };
  const CUtensorMap m0 = map(a[0], OM);
  oz_launch<kOzGram>(dim3((int)splits, tiles), m0, segs > 1 ? map(a[1], OM) : m0,
                     map(b, ON), g, s);
  sum_splits(partials, (int)splits, count, out, s);
}

static void oz_product(const OzBlock& a, int k, int n, const double* M,
                       const OzSmall& w, OzArgs g, bool grad, int* grid_out,
                       cudaStream_t s) {
  const int ldk = oz_ldk(k);
  auto* dig = static_cast<__nv_bfloat16*>(w.digits);
  k_oz_slice_small<<<n, 128, 0, s>>>(k, ldk, M, a.scale, dig, w.scale);
  TRM_CHECK_LAUNCH();
  const int64_t lds = oz_ld(a.N);
  g.N = a.N;
  g.m = k;
  g.n = n;
  g.tiles_m = ceil_div(a.N, (int64_t)OM);
  g.tiles_n = ceil_div(n, ON);
  g.sb = w.scale;
  const CUtensorMap ma = oz_map(static_cast<const __nv_bfloat16*>(a.digits), lds,
                                a.m, lds, lds * a.m, 64, OK, true);
  const CUtensorMap mb = oz_map(dig, k, n, ldk, (int64_t)ldk * n, OK, ON, false);
  const int grid = oz_product_parts(a.N, n);
  if (grad)
    oz_launch<kOzGrad>(dim3(grid), ma, ma, mb, g, s);
  else
    oz_launch<kOzStore>(dim3(grid), ma, ma, mb, g, s);
  if (grid_out) *grid_out = grid;
}

int oz_product_parts(int64_t N, int n) {
  return (int)std::min<int64_t>(
      sm_count(), (int64_t)ceil_div(N, (int64_t)OM) * ceil_div(n, ON));
}

void oz_mult(const OzBlock& a, int n, const double* M, bool tri,
             const OzSmall& w, double* Y, int64_t ldy, int* err,
             cudaStream_t s, const int* halt) {
  OzArgs g{};
  g.halt = halt;
  g.out = Y;
  g.ldo = ldy;
  g.tri = tri ? 1 : 0;
  g.err = err;
  oz_product(a, a.m, n, M, w, g, false, nullptr, s);
}

void oz_grad(const OzBlock& a, const double* Hp, const OzSmall& w,
             const double* Xp, double* G, const double* Gprev,
             const double* Pprev, const double* minv, int64_t ld, double* part,
             IterScalars* sc, cudaStream_t s) {
  OzArgs g{};
  g.out = G;
  g.ldo = ld;
  g.xp = Xp;
  g.gprev = Gprev;
  g.pprev = Pprev;
  g.minv = minv;
  g.part = part;
  g.err = &sc->status;
  int grid = 0;
  oz_product(a, a.m, a.m, Hp, w, g, true, &grid, s);
  cg_from_parts(part, grid, a.m, sc, s);
}

}  // namespace trm
