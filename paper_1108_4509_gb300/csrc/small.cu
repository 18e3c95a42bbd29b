// m x m matrix work on the device: products, the line model along P,
// Cholesky factorisation and triangular inverse (Fig. ONFIG steps (2), (3)),
// and the symmetric eigenproblem of the closing Rayleigh-Ritz step
// (Sec. 2.1: "diagonalization of H ... will give the explicit eigenvalues").
// All matrices are column-major with leading dimension m and stored as FP64;
// the template parameter Tm is the arithmetic type.
#include <atomic>
#include <cstdlib>

#include "dfmath.cuh"
#include "ops.cuh"
#include "tc.cuh"

namespace trm {

namespace {

// ---------------------------------------------------------------------------
// Cm = alpha op(A) op(B) + beta Cin, 8 x 8 tiles on 256 threads: four threads
// share an output, each a quarter of every 64-deep stage, in two chains. An
// SM does two FP64 multiply-adds a cycle, so these matrices are spread over as
// many SMs as they fill: 4.9 us at m = 48, 5.6 at 64, 8.3 at 128, 35 at 256
// with launches back to back; 16 x 16 tiles, one thread per output, take 8.2,
// 8.3, 14 and 41 (m = 512: 231 and 238, m = 1024: 1780 and 1762).
//
// skip (may be null): when *skip is below kNsDone the product is not formed
// and Cm becomes a copy of Cin (is left alone without one). dev (may be null):
// receives max |Cm - I|, as the bits of a non-negative double.
// ---------------------------------------------------------------------------
// A Newton-Schulz step takes X^T X - I = E to 3/4 E^2 + 1/4 E^3: from entries
// below 1e-10 to below m 1e-20, less than rounding leaves, so the steps after
// that one change nothing.
constexpr double kNsDone = 1e-10;

// Acceptance of chol_refined's result: max |X S X^T - I| after one correction
// (another then leaves m 1e-20), max |X - I| after both, and no kernel before
// them that saw the attempt to be in vain (dev[kRefStop]).
enum { kRefDev1 = 1, kRefDev2 = 2, kRefStop = 3, kRefWords = 4 };
__device__ __forceinline__ bool refined_ok(const unsigned long long* dev) {
  return dev[kRefStop] == 0ull &&
         __longlong_as_double((long long)dev[kRefDev1]) < 1e-10 &&
         __longlong_as_double((long long)dev[kRefDev2]) < 0.5;
}

// tri: which operands are lower triangular (the products then leave out what
// lies beyond their tiles), and Phi: 1 where only the lower triangle of
// Cm - I is wanted, with half its diagonal (dev as before).
enum { kTriA = 1, kTriB = 2, kTriBt = 4, kTriOut = 8, kPhi = 16 };

struct GemmOpt {
  const double* cin = nullptr;
  const unsigned long long* skip = nullptr;
  const unsigned long long* stop = nullptr;  // not null: nothing when not 0
  unsigned long long* dev = nullptr;
  int tri = 0;
};

__global__ void __launch_bounds__(256)
    k_mm_gemm(int m, const double* __restrict__ A, int trA,
              const double* __restrict__ B, int trB, double* __restrict__ Cm,
              double alpha, double beta, GemmOpt opt) {
  constexpr int TT = 8;   // tile
  constexpr int KS = 4;   // threads per output
  constexpr int KD = 64;  // stage depth
  __shared__ double As[KD][TT + 1], Bs[KD][TT + 1];
  __shared__ double part[KS][TT * TT];
  const int tid = threadIdx.x;
  const int o = tid % (TT * TT), ks = tid / (TT * TT);
  const int tx = o % TT, ty = o / TT;
  const int i0 = blockIdx.x * TT, j0 = blockIdx.y * TT;
  const int i = i0 + tx, j = j0 + ty;
  const bool in = i < m && j < m;
  const int64_t e = i + (int64_t)j * m;
  if (opt.skip && __longlong_as_double((long long)*opt.skip) < kNsDone) {
    if (in && ks == 0 && opt.cin) Cm[e] = opt.cin[e];
    return;
  }
  if (opt.stop && *opt.stop) return;
  if ((opt.tri & kTriOut) && j0 > i0) return;
  int kb = 0, ke = m;  // the sum's range
  if (opt.tri & kTriA) ke = min(ke, i0 + TT);
  if (opt.tri & kTriBt) ke = min(ke, j0 + TT);
  if (opt.tri & kTriB) kb = j0;
  double a0 = 0.0, a1 = 0.0;
  for (int k0 = kb; k0 < ke; k0 += KD) {
    for (int q = tid; q < KD * TT; q += 256) {
      // each operand along its contiguous index
      const int kr = trA ? q % KD : q / TT, r = trA ? q / KD : q % TT;
      As[kr][r] = (i0 + r < m && k0 + kr < ke)
                      ? (trA ? A[(k0 + kr) + (int64_t)(i0 + r) * m]
                             : A[(i0 + r) + (int64_t)(k0 + kr) * m])
                      : 0.0;
      const int kc = trB ? q / TT : q % KD, c = trB ? q % TT : q / KD;
      Bs[kc][c] = (k0 + kc < ke && j0 + c < m)
                      ? (trB ? B[(j0 + c) + (int64_t)(k0 + kc) * m]
                             : B[(k0 + kc) + (int64_t)(j0 + c) * m])
                      : 0.0;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 16; k += 2) {
      a0 = fma(As[16 * ks + k][tx], Bs[16 * ks + k][ty], a0);
      a1 = fma(As[16 * ks + k + 1][tx], Bs[16 * ks + k + 1][ty], a1);
    }
    __syncthreads();
  }
  double acc = a0 + a1;
  part[ks][o] = acc;
  __syncthreads();
  if (ks == 0)
#pragma unroll
    for (int q = 1; q < KS; ++q) acc += part[q][o];
  double d = 0.0;
  if (in && ks == 0) {
    const double v = alpha * acc + (beta != 0.0 ? beta * opt.cin[e] : 0.0);
    d = v - (i == j ? 1.0 : 0.0);
    Cm[e] = !(opt.tri & kPhi) ? v : i > j ? d : i == j ? 0.5 * d : 0.0;
  }
  if (opt.dev) {
    // (a NaN's bits are above every number's: it never reads as converged)
    unsigned long long b = (unsigned long long)__double_as_longlong(fabs(d));
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) {
      const unsigned long long x = __shfl_xor_sync(0xffffffffu, b, s);
      b = x > b ? x : b;
    }
    if ((tid & 31) == 0 && b) atomicMax(opt.dev, b);
  }
}

static void mm_launch(int m, const double* A, bool trA, const double* B, bool trB,
                      double* Cm, double alpha, double beta, const GemmOpt& opt,
                      cudaStream_t s) {
  const int t = ceil_div(m, 8);
  k_mm_gemm<<<dim3(t, t), 256, 0, s>>>(m, A, trA, B, trB, Cm, alpha, beta, opt);
  TRM_CHECK_LAUNCH();
}

// A0 = sym(H') + diag(H_D): the projected matrix C^T H C when C^T C = I
// (H_D may be null: plain symmetrisation).
__global__ void k_make_A0(int m, const double* __restrict__ Hp,
                          const double* __restrict__ HD, double* A0) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= (int64_t)m * m) return;
  const int i = (int)(e % m), j = (int)(e / m);
  double v = 0.5 * (Hp[i + (int64_t)j * m] + Hp[j + (int64_t)i * m]);
  if (i == j && HD) v += HD[i];
  A0[e] = v;
}

// ---------------------------------------------------------------------------
// Line model along P. With R = H C - C A0 = -G/2, the block pencil C + a P
// (C^T C = I) has S(a) = I + a S1 + a^2 Q and A(a) - S(a) A0 = a D1 + a^2 D2,
//   S1 = B + B^T,  D1 = A0 B - B A0 - (W + W^T)/2,  D2 = P^T H P - Q A0,
// with B = C^T P, Q = P^T P, W = P^T G. Every term is formed from small
// quantities, so E(a) - E(0) = tr(S(a)^{-1} (a D1 + a^2 D2)) keeps its
// relative accuracy close to convergence. To second order
//   E(a) - E(0) = a tr(D1) + a^2 (tr(D2) - tr(S1 D1)).
// ---------------------------------------------------------------------------

// Reciprocal square root and reciprocal of the pivot chain by Newton's
// method from the hardware approximations (rsqrt, reciprocal): one step in
// FP32, two from the FP32 seed in FP64. Arguments are positive normal numbers (the pivot
// tests come first); the results are within a few ulp, and the chain stays
// free of the slow-path calls of the IEEE operations.
__device__ __forceinline__ float piv_rcp(float t) {
  const float r = __fdividef(1.0f, t);
  return fmaf(r, fmaf(-t, r, 1.0f), r);
}
__device__ __forceinline__ double piv_rcp(double t) {
  double r = (double)__fdividef(1.0f, (float)t);
  r = fma(r, fma(-t, r, 1.0), r);
  return fma(r, fma(-t, r, 1.0), r);
}
// 1 / sqrt(t): the hardware reciprocal square root refined by Newton's step
// r <- r (3 - t r^2) / 2, once in FP32, twice (from the FP32 seed) in FP64.
__device__ __forceinline__ float piv_rsqrt(float t) {
  const float r = rsqrtf(t);
  return r * fmaf(-0.5f * t * r, r, 1.5f);
}
__device__ __forceinline__ double piv_rsqrt(double t) {
  double r = (double)rsqrtf((float)t);
  r = r * fma(-0.5 * t * r, r, 1.5);
  return r * fma(-0.5 * t * r, r, 1.5);
}

// The step along P: minimiser of the parabola a tr(D1) + a^2 (tr(D2) -
// tr(S1 D1)), bounded so that the RMS column change a ||P||_F / sqrt(m)
// stays below 1; a restart is requested when P is not a descent direction.
// (One division by Newton's method where the FP32 seed is in range, and the
// cap's square root only where the cap binds: the FP64 library calls of this
// chain cost more than the sums before it.)
__device__ __forceinline__ double line_alpha(int m, const double* v,
                                             const IterScalars* sc) {
  const double g0 = v[0];
  const double c2 = v[1] - v[2];
  const double qn = v[3];
  if (!(g0 < 0.0 && qn > 0.0)) return 0.0;
  double alpha;
  if (c2 > 1e-30 && c2 < 1e30)
    alpha = -0.5 * g0 * piv_rcp(c2);
  else if (c2 > 0.0)
    alpha = -g0 / (2.0 * c2);
  else
    alpha = sc->alpha_prev > 0.0 ? 2.0 * sc->alpha_prev
                                 : 0.5 * sqrt((double)m / qn);
  if (!(alpha * alpha * qn <= (double)m)) alpha = sqrt((double)m / qn);
  return alpha;
}
// What the step leaves in sc (after every reader of alpha_prev).
__device__ __forceinline__ void line_store(const double* v, double alpha,
                                           IterScalars* sc) {
  const double g0 = v[0], c2 = v[1] - v[2];
  if (!(g0 < 0.0 && v[3] > 0.0))
    sc->restart = 1;  // not a descent direction: restart CG next time
  sc->alpha = alpha;
  if (alpha > 0.0) sc->alpha_prev = alpha;
  sc->c2 = c2;
  sc->dE = alpha * g0 + alpha * alpha * c2;
}
__device__ void line_alpha_block(int m, const double* __restrict__ part,
                                 int nparts, IterScalars* sc, double* red) {
  double v[4] = {0, 0, 0, 0};
  for (int p = threadIdx.x; p < nparts; p += blockDim.x)
#pragma unroll
    for (int q = 0; q < 4; ++q) v[q] += part[(size_t)p * 4 + q];
  block_sum4(v, red);
  if (threadIdx.x == 0) line_store(v, line_alpha(m, v, sc), sc);
}

// ---------------------------------------------------------------------------
// FP64 Cholesky S = L L^T and L^{-1}, blocked in 32-column panels, one CTA of 256
// threads. Writes Linv (lower) and R = L^{-T} (upper).
//
// m is padded to mp, a multiple of 32, with the identity, which changes
// neither factor. Per panel p: (a) the eight warps factor the diagonal block
// column by column (right-looking), four columns per warp in registers: the
// owner of a column takes its pivot by a shuffle and publishes the column
// through shared memory, and each warp updates its own columns; (b) every row
// below solves x L_pp^T = a (registers, reciprocal pivots from (a));
// (c) all threads update the lower trailing triangle with 4 x 4 register
// tiles. The inverse: (d) warp p inverts diagonal block p by forward
// substitution, one column of the inverse per lane in registers, rows of L
// read as broadcasts; (e) row-block by row-block,
// X_ij = -X_ii sum_{k=j}^{i-1} L_ik X_kj through a 32 x mp temporary. The
// working copy has leading dimension mp + 1. Linv may be null (only R is
// written then). Every pivot chain step is a dependent sequence, so the
// phases avoid shuffles and global loads inside it.
//
// S is read from memory, or (Bm != null) formed on the fly as
// S = I + a (B + B^T) + a^2 Q with a = sc->alpha (the line step's overlap).
//
// With dev = true the other kernels here run in deviation form for S = I + E:
// L = I + F and L^{-1} = I + Y with the identity kept exact and only the
// small E, F, Y held. Pivot: d = E_cc - sum_k F_ck^2 and
// f_cc = d / (1 + sqrt(1 + d)); off the diagonal L and F coincide; inverse
// diagonal y_cc = -f_cc / (1 + f_cc). When S - I is small, FP32 arithmetic
// here yields L to FP64 accuracy relative to I.
// ---------------------------------------------------------------------------
// Cholesky of a 32 x 32 diagonal block on one warp (Fig. ONFIG step (2)
// restricted to the block). Lane r holds row r of the block in w (w[j] =
// entry (r, j), meaningful for j <= r) and ends with row r of L (of F in
// deviation form, L = I + F); rd[c] = 1 / L_cc. The pivot of column c comes
// from lane c by a shuffle and the entries L_jc (j > c) of the rank-1 update
// from lanes j, so the 32 steps need no barrier. Entries above the diagonal
// are updated too and never read. thr: the pivot floor of column `lane`
// (plain form). Returns true when a pivot was not positive (singular S).
// Used by the blocked factorisation's diagonal kernel; the single-CTA
// kernel keeps its eight-warp column steps, which measured faster there
// (10.5K against 12.3K cycles per 32-column panel at m = 128: one warp
// issues all 31 - c shuffles of a step by itself).
template <typename Tm, bool dev>
__device__ __forceinline__ bool diag_factor_warp(Tm (&w)[32], Tm thr, Tm* rd) {
  const int lane = threadIdx.x & 31;
  bool b = false;
#pragma unroll
  for (int c = 0; c < 32; ++c) {
    Tm d = __shfl_sync(0xffffffffu, w[c], c);
    Tm rl;
    if (dev) {
      if (!(d > (Tm)-0.999)) {  // pivot 1 + d not positive
        b = true;
        d = (Tm)0;
      }
      rl = piv_rsqrt((Tm)1 + d);
    } else {
      if (!(d > __shfl_sync(0xffffffffu, thr, c))) {
        b = true;
        d = (Tm)1;
      }
      rl = piv_rsqrt(d);
    }
    const Tm l = lane > c ? w[c] * rl : w[c];  // L_rc for r > c
    if (lane == 0) rd[c] = rl;
    // L_cc (deviation form: L_cc - 1 = d / (1 + sqrt(1 + d)), with
    // sqrt(1 + d) = (1 + d) rl, which keeps small d accurate)
    w[c] = lane == c ? (dev ? d * piv_rcp((Tm)1 + ((Tm)1 + d) * rl) : d * rl)
                     : l;
#pragma unroll
    for (int j = c + 1; j < 32; ++j) w[j] -= l * __shfl_sync(0xffffffffu, l, j);
  }
  return b;
}

// X = L^{-1} of a 32 x 32 lower-triangular diagonal block (Fig. ONFIG step
// (3) restricted to the block): L in shared memory at B[i + k ldb], rd[i] =
// 1 / L_ii. Lane j forms column j of X in x by forward substitution,
// x_ij = (delta_ij - sum_{k=j}^{i-1} L_ik x_kj) / L_ii, with the column in
// registers and the rows of L read as broadcasts (x_kj = 0 for k < j, so
// the sums run over all k < i). Deviation form (L = I + F, X = I + Y):
// y_jj = -f_jj / (1 + f_jj), y_ij = -(f_ij + sum_k f_ik y_kj) / (1 + f_ii).
template <typename Tm, bool dev>
__device__ __forceinline__ void diag_inverse_warp(const Tm* B, int ldb,
                                                  const Tm* rd, Tm (&x)[32]) {
  const int j = threadIdx.x & 31;
#pragma unroll
  for (int i = 0; i < 32; ++i) {
    Tm s0 = (dev && i > j) ? B[i + j * ldb] : (Tm)0, s1 = 0;
#pragma unroll
    for (int k = 0; k < i; ++k) {
      if (k & 1) s1 += B[i + k * ldb] * x[k];
      else s0 += B[i + k * ldb] * x[k];
    }
    const Tm r = rd[i];
    x[i] = i == j ? (dev ? -B[i + i * ldb] * r : r)
                  : (i > j ? -(s0 + s1) * r : (Tm)0);
  }
}

// 256 threads: the register-resident rows of the diagonal-block steps need
// more than the 128 registers a 512-thread CTA allows (they spilled, and
// the sequential pivot chain paid for it); the parallel phases lose less.
constexpr int kCholThreads = 256;

// SM: the working copy lives in shared memory (a compile-time choice, so its
// accesses compile to shared-memory instructions), else in gwork.
template <bool SM>
__global__ void __launch_bounds__(kCholThreads, 1)
    k_chol_inv(int m, const double* __restrict__ S, const double* __restrict__ Bm,
               const double* __restrict__ Q, double* __restrict__ Linv,
               double* __restrict__ R, IterScalars* sc, double* gwork,
               const double* __restrict__ lpart, int nlpart,
               const unsigned long long* refined) {
  if (refined && refined_ok(refined)) return;
  using Tm = double;
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ int bad;
  __shared__ Tm rdiag[1024];  // 1 / L_cc, all columns (mp <= 1024)
  const int tid = threadIdx.x, nt = blockDim.x;
  const int lane = tid & 31, warp = tid >> 5, nw = nt >> 5;
  const int mp = (m + 31) & ~31, ld = mp + 1, P = mp >> 5;
  Tm* a = SM ? reinterpret_cast<Tm*>(smraw) : gwork;
  Tm* tb = a + (size_t)mp * ld;  // 32 x mp, leading dimension 33
  const Tm eps = 2.3e-16;
  if (lpart) {  // the line step first (it sets sc->alpha)
    __shared__ double lred[4 * 32];
    line_alpha_block(m, lpart, nlpart, sc, lred);
    __syncthreads();
  }
  if (Bm) {
    // half of a (B + B^T) + a^2/2 (Q + Q^T) from each triangle, read in
    // column order (four loads of each matrix in flight per thread), then
    // the lower triangle adds its mirror.
    const double al = sc->alpha;
    const double hq = 0.5 * al * al;
    for (int k = warp; k < mp; k += nw)
      for (int i0 = lane; i0 < mp; i0 += 128) {
        Tm t[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int i = i0 + 32 * u;
          const bool in = i < m && k < m;
          t[u] = in ? (Tm)(al * Bm[i + k * m] + hq * Q[i + k * m]) : (Tm)0;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (i0 + 32 * u < mp) a[(i0 + 32 * u) + k * ld] = t[u];
      }
    __syncthreads();
    for (int k = warp; k < mp; k += nw)
      for (int i = k + lane; i < mp; i += 32)
        a[i + k * ld] = a[i + k * ld] + a[k + i * ld] + (i == k ? 1.0 : 0.0);
  } else {
    for (int k = warp; k < mp; k += nw)
      for (int i = k + lane; i < mp; i += 32) {
        a[i + k * ld] = i < m && k < m ? S[i + k * m] : i == k ? 1.0 : 0.0;
      }
  }
  if (tid == 0) bad = 0;
  __syncthreads();

  for (int p = 0; p < P; ++p) {
    const int c0 = 32 * p;
    // (a) diagonal block on all eight warps: warp w keeps columns w, w + 8,
    // w + 16 and w + 24 of the block in registers (lane r = row c0 + r).
    // For column c the owning warp forms the pivot and publishes the column
    // through shared memory (two buffers, so one barrier per column); every
    // warp then updates its own later columns. Lanes above the diagonal
    // update too: those entries are never read.
    {
      __shared__ Tm colbuf[2][32];
      const int r = c0 + lane;
      Tm v[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) v[q] = a[r + (c0 + warp + 8 * q) * ld];
      bool b = false;
#pragma unroll
      for (int c = 0; c < 32; ++c) {
        const int q = c >> 3;
        if (warp == (c & 7)) {
          Tm d = __shfl_sync(0xffffffffu, v[q], c);
          // 1 / L_cc is all the column needs: rsqrt(d) on the pivot chain; L_cc
          // itself is formed after the column is out
          // a pivot that has lost all but 4m roundings of its original
          // diagonal entry marks a (numerically) singular S
          const int cc = c0 + c;
          const double sjj = (Bm || cc >= m) ? 1.0 : fabs(S[cc + cc * m]);
          if (!(d > (Tm)(4 * m) * eps * sjj)) {
            b = true;
            d = 1.0;
          }
          const Tm rl = piv_rsqrt(d);
          if (lane > c) v[q] *= rl;
          colbuf[c & 1][lane] = v[q];  // the diagonal entry is not read
          if (lane == 0) rdiag[c0 + c] = rl;
          if (lane == c) v[q] = d * rl;
        }
        __syncthreads();
        const Tm lrc = colbuf[c & 1][lane];
#pragma unroll
        for (int qq = 0; qq < 4; ++qq)
          if (warp + 8 * qq > c) v[qq] -= lrc * colbuf[c & 1][warp + 8 * qq];
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) a[r + (c0 + warp + 8 * q) * ld] = v[q];
      if (lane == 0 && b) bad = 1;
    }
    __syncthreads();
    // (b) rows below the block: x L_pp^T = a
    for (int r = c0 + 32 + tid; r < mp; r += nt) {
      Tm x[32];
#pragma unroll
      for (int c = 0; c < 32; ++c) x[c] = a[r + (c0 + c) * ld];
#pragma unroll
      for (int c = 0; c < 32; ++c) {
        Tm s0 = x[c], s1 = 0;
#pragma unroll
        for (int k = 0; k < 31; k += 2) {
          if (k < c) s0 -= x[k] * a[(c0 + c) + (c0 + k) * ld];
          if (k + 1 < c) s1 -= x[k + 1] * a[(c0 + c) + (c0 + k + 1) * ld];
        }
        x[c] = (s0 + s1) * rdiag[c0 + c];
      }
#pragma unroll
      for (int c = 0; c < 32; ++c) a[r + (c0 + c) * ld] = x[c];
    }
    __syncthreads();
    // (c) lower trailing triangle, 4 x 4 tiles
    const int base = c0 + 32;
    const int T = (mp - base) >> 2;
    const int ntile = T * (T + 1) / 2;
    for (int t = tid; t < ntile; t += nt) {
      int ti = (int)((sqrtf(8.0f * t + 1.0f) - 1.0f) * 0.5f);
      while ((ti + 1) * (ti + 2) / 2 <= t) ++ti;
      while (ti * (ti + 1) / 2 > t) --ti;
      const int tj = t - ti * (ti + 1) / 2;
      const int r0 = base + 4 * ti, s0 = base + 4 * tj;
      Tm acc[4][4] = {};
#pragma unroll 8
      for (int k = 0; k < 32; ++k) {
        Tm lr[4], ls[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          lr[u] = a[(r0 + u) + (c0 + k) * ld];
          ls[u] = a[(s0 + u) + (c0 + k) * ld];
        }
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
          for (int v = 0; v < 4; ++v) acc[u][v] += lr[u] * ls[v];
      }
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v)
          if (r0 + u >= s0 + v) a[(r0 + u) + (s0 + v) * ld] -= acc[u][v];
    }
    __syncthreads();
  }

  // (d) inverse X = L_pp^{-1} of each diagonal block, one warp per block,
  // in place, row by row: lane j forms X_ij = (delta_ij - sum_{k=j}^{i-1}
  // L_ik X_kj) / L_ii from row i of L and its own column of X (rolled loops:
  // code run once per launch would stall on instruction fetch).
  for (int pb = warp; pb < P; pb += nw) {
    Tm* B = a + 32 * pb + (size_t)(32 * pb) * ld;  // block (i, k) at B[i + k ld]
    const Tm* rd = rdiag + 32 * pb;
    const int j = lane;
    for (int i = 0; i < 32; ++i) {
      Tm s0 = 0, s1 = 0;
      int k = j;
#pragma unroll 2
      for (; k + 1 < i; k += 2) {
        s0 += B[i + k * ld] * B[k + j * ld];
        s1 += B[i + (k + 1) * ld] * B[(k + 1) + j * ld];
      }
      if (k < i) s0 += B[i + k * ld] * B[k + j * ld];
      Tm x = 0;
      if (i == j) x = rd[i];
      else if (i > j) x = -(s0 + s1) * rd[i];
      __syncwarp();  // row i of L is read by every lane before it is replaced
      if (i >= j) B[i + j * ld] = x;
      __syncwarp();
    }
  }
  __syncthreads();
  // (e) off-diagonal blocks, row-block by row-block: T = L_{i,0:i} X_{0:i,0:i}
  // (32 x ri, through tb), then X_{i,0:i} = -X_ii T; 4 x 4 register tiles.
  // Only the lower triangle of the working copy is read.
  for (int i = 1; i < P; ++i) {
    const int ri = 32 * i;
    const int nblk = 2 * ri;  // 8 row groups x ri/4 column groups
    for (int bq = tid; bq < nblk; bq += nt) {
      const int r0 = 4 * (bq & 7), cb = 4 * (bq >> 3);
      Tm acc[4][4] = {};
#pragma unroll 4
      for (int col = cb; col < ri; ++col) {
        Tm lr[4], xc[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) lr[u] = a[(ri + r0 + u) + col * ld];
#pragma unroll
        for (int v = 0; v < 4; ++v)
          xc[v] = col >= cb + v ? a[col + (cb + v) * ld] : (Tm)0;
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
          for (int v = 0; v < 4; ++v) acc[u][v] += lr[u] * xc[v];
      }
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v) tb[(r0 + u) + (cb + v) * 33] = acc[u][v];
    }
    __syncthreads();
    for (int bq = tid; bq < nblk; bq += nt) {
      const int r0 = 4 * (bq & 7), cb = 4 * (bq >> 3);
      Tm acc[4][4] = {};
#pragma unroll 4
      for (int q = 0; q <= r0 + 3; ++q) {
        Tm xr[4], tv[4];
#pragma unroll
        for (int u = 0; u < 4; ++u)
          xr[u] = q <= r0 + u ? a[(ri + r0 + u) + (ri + q) * ld] : (Tm)0;
#pragma unroll
        for (int v = 0; v < 4; ++v) tv[v] = tb[q + (cb + v) * 33];
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
          for (int v = 0; v < 4; ++v) acc[u][v] += xr[u] * tv[v];
      }
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 4; ++v) a[(ri + r0 + u) + (cb + v) * ld] = -acc[u][v];
    }
    __syncthreads();
  }
  const int isbad = bad;
  // Linv(i, k) column by column, then R(k, i) = Linv(i, k) column by column,
  // four entries per thread in flight
  auto entry = [&](int i, int k) -> double {
    if (isbad) return i == k ? 1.0 : 0.0;
    return i >= k ? a[i + k * ld] : 0.0;
  };
  for (int o = 0; o < (Linv ? 2 : 1); ++o) {
    double* out = o ? Linv : R;
    for (int k = warp; k < m; k += nw)  // column k of Linv, row k of R
      for (int i0 = lane; i0 < m; i0 += 128) {
        double v[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int i = i0 + 32 * u;
          v[u] = i < m ? (o ? entry(i, k) : entry(k, i)) : 0.0;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int i = i0 + 32 * u;
          if (i < m) out[i + k * m] = v[u];
        }
      }
  }
  if (tid == 0 && isbad && sc) sc->status |= 1;
}

// ---------------------------------------------------------------------------
// The FP32 factorisation for m <= 256: S = L L^T and X = L^{-1} in one CTA of
// 16 warps, by block elimination on [S | I] with 32-column panels. The working
// copy M holds the lower 32 x 32 blocks (row-major, leading dimension 36) in
// shared memory; block (i, j) starts as A_ij and turns, once panel j has been
// eliminated, into the block W_ij of the growing inverse, so no other copy of
// either triangle exists. Panel p:
//   (1) warp 0 factors the diagonal block, one row per lane in registers;
//       warp 1 follows one group of four columns behind and forms
//       X_pp = L_pp^{-1}, one column per lane;
//   (2) Z (32 x mp) takes what this panel contributes to every block column:
//       X_pj = X_pp W_pj for j < p, X_pp, and L_ip = A_ip X_pp^T for i > p;
//   (3) every block (i, j), i > p, j <= i, takes M_ij -= L_ip Z_j, with M_ip
//       starting from zero: the Cholesky update for j > p and the inverse's
//       for j <= p are the same product, 8 x 4 register tiles. Four warps
//       update the next diagonal block first and two go on with (1) for it,
//       so the pivot chain runs beside the updates.
// What bounds it is that chain (one dependent rsqrt, multiply, shuffle per
// column, about 110 cycles) and one SM's FP32 rate: 38 us at m = 128 and 86 at
// 220 from cold caches, where a kernel with separate factor, solve and inverse
// phases took 78 and 376. In deviation form (dev,
// S = I + E, see above) only the diagonal needs care: it holds the deviation
// d of the pivot from 1, and y_cc = -f_cc / L_cc is kept apart (ydiag).
// With `split` the inverse goes out as the two TF32 terms the product kernels
// read (hi, lo, leading dimension ldm, the part below the diagonal left as it
// is; split_diag: the diagonal zero and written as FP32 pairs after them), else
// as FP64 R = L^{-T}.
// ---------------------------------------------------------------------------
constexpr int PLD = 36, PSZ = 32 * PLD;  // block row stride, block size
constexpr int kPanelMax = 256;
constexpr int kPanelThreads = 512;

__host__ __device__ constexpr int panel_blocks(int P) { return P * (P + 1) / 2; }
inline size_t panel_smem(int m) {
  const int P = (m + 31) >> 5;
  return ((size_t)panel_blocks(P) * PSZ + (size_t)32 * (32 * P + 4) +
          33 * 32 + 32) * sizeof(float);
}

// 1 / sqrt(t), t a positive normal number: one instruction and a Newton step
// (piv_rsqrt without the library call's subnormal path).
__device__ __forceinline__ float panel_rsqrt(float t) {
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(t));
  return r * fmaf(-0.5f * t * r, r, 1.5f);
}

// Factor the diagonal block D (warp 0; the updated block in shared memory).
// lcol[c][r] = L_rc (0 for r <= c), rd[c] = 1 / L_cc, ydg[c] = y_cc. Four
// columns a round: within it only the round's own columns are updated, by
// shuffles; the other columns take the round's rank-4 update from shared memory
// during the next one, in the shadow of its pivot chain (shuffle, rsqrt with a
// Newton step, two multiplies: about 100 of the 180 cycles a column takes). The
// row moves down by four registers a round, so that every index is static and
// the code is short. thr: pivot floor of column `lane`.
template <bool dev>
__device__ __forceinline__ bool panel_factor(const float* D, float thr,
                                             float* lcol, float* rd,
                                             float* ydg) {
  const int lane = threadIdx.x & 31;
  float w[32];
#pragma unroll
  for (int j = 0; j < 32; j += 4) {
    const float4 t = *reinterpret_cast<const float4*>(D + lane * PLD + j);
    w[j] = t.x; w[j + 1] = t.y; w[j + 2] = t.z; w[j + 3] = t.w;
  }
  bool bad = false;
  float dk = 0.f, rk = 1.f;  // pivot and 1 / L_cc of this lane's column
  float lp[4] = {0.f, 0.f, 0.f, 0.f};  // the round before: its column entries
  float dn = w[0];  // in lane c: the pivot of column c
#pragma unroll 1
  for (int g = 0; g < 8; ++g) {
    float l[4];
    const float* lv = lcol + 132 * g;   // column 4 g from row 4 g on
    const float* pv = g ? lv - 128 : lv;  // the round before, from row 4 g on
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int c = 4 * g + u;
      // (a pivot that is not positive makes everything after it meaningless;
      // the caller then writes the identity)
      const float d = __shfl_sync(0xffffffffu, dn, c);
      const float t = dev ? 1.f + d : d;  // the pivot
      bad |= !(d > (dev ? -0.999f : __shfl_sync(0xffffffffu, thr, c)));
      const float rl = panel_rsqrt(t);
      l[u] = lane > c ? w[u] * rl : 0.f;
      // the next pivot: its lane has the row's entries itself, so the chain
      // does not wait for the column's broadcast
      if (u < 3) {
        dn = w[u + 1] - l[u] * l[u];
      } else {
        dn = w[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) dn -= l[e] * l[e];
      }
#pragma unroll
      for (int v = u + 1; v < 4; ++v)
        w[v] -= l[u] * __shfl_sync(0xffffffffu, l[u], 4 * g + v);
      if (lane == c) {
        dk = d;
        rk = rl;
      }
      // the update by the round before, a quarter of it in each column's
      // shadow (lp = 0 in the first round, where pv reads unwritten entries)
      if (g) {
#pragma unroll
        for (int q = 1 + 2 * u; q < 3 + 2 * u && q < 8; ++q)
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const float4 b =
                *reinterpret_cast<const float4*>(pv + 32 * e + 4 * q);
            w[4 * q + 0] -= lp[e] * b.x;
            w[4 * q + 1] -= lp[e] * b.y;
            w[4 * q + 2] -= lp[e] * b.z;
            w[4 * q + 3] -= lp[e] * b.w;
          }
      }
      lcol[32 * c + lane] = l[u];
      if (lane == 0) rd[c] = rl;
    }
    __syncwarp();
    // columns 4 g .. 4 g + 3 are out: warp 1 may use them
    asm volatile("bar.arrive %0, 64;" ::"r"(1 + g) : "memory");
    // the next round's own columns now, the others in its shadow
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const float4 b = *reinterpret_cast<const float4*>(lv + 32 * e + 4);
      w[4] -= l[e] * b.x;
      w[5] -= l[e] * b.y;
      w[6] -= l[e] * b.z;
      w[7] -= l[e] * b.w;
      lp[e] = l[e];
    }
#pragma unroll
    for (int j = 0; j < 28; ++j) w[j] = w[j + 4];
  }
  // L_cc - 1 = d / (1 + sqrt(1 + d)) with sqrt(1 + d) = (1 + d) rl
  if (dev) ydg[lane] = -(dk * piv_rcp(1.f + (1.f + dk) * rk)) * rk;
  return bad;
}

// X = L^{-1} of the diagonal block into D (warp 1, a round behind warp 0):
// lane j runs column j of the forward substitution, right-looking.
__device__ __forceinline__ void panel_invert(float* D, const float* lcol,
                                             const float* rd) {
  const int lane = threadIdx.x & 31;
  float a[32];
#pragma unroll
  for (int i = 0; i < 32; ++i) a[i] = i == lane ? 1.f : 0.f;
#pragma unroll 1
  for (int g = 0; g < 8; ++g) {
    asm volatile("bar.sync %0, 64;" ::"r"(1 + g) : "memory");
    const float* lv = lcol + 132 * g;
    const float4 r4 = *reinterpret_cast<const float4*>(rd + 4 * g);
    const float4 l0 = *reinterpret_cast<const float4*>(lv);
    const float4 l1 = *reinterpret_cast<const float4*>(lv + 32);
    const float4 l2 = *reinterpret_cast<const float4*>(lv + 64);
    float x[4];
    x[0] = a[0] * r4.x;
    x[1] = (a[1] - l0.y * x[0]) * r4.y;
    x[2] = (a[2] - l0.z * x[0] - l1.z * x[1]) * r4.z;
    x[3] = (a[3] - l0.w * x[0] - l1.w * x[1] - l2.w * x[2]) * r4.w;
#pragma unroll
    for (int u = 0; u < 4; ++u) D[(4 * g + u) * PLD + lane] = x[u];
#pragma unroll
    for (int q = 1; q < 8; ++q) {
      float4 b[4];
#pragma unroll
      for (int u = 0; u < 4; ++u)
        b[u] = *reinterpret_cast<const float4*>(lv + 32 * u + 4 * q);
      const int o = 4 * q - 4;
      a[o + 0] = a[o + 4];
      a[o + 1] = a[o + 5];
      a[o + 2] = a[o + 6];
      a[o + 3] = a[o + 7];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        a[o + 0] -= b[u].x * x[u];
        a[o + 1] -= b[u].y * x[u];
        a[o + 2] -= b[u].z * x[u];
        a[o + 3] -= b[u].w * x[u];
      }
    }
  }
}

// M_ij -= L_ip Z_j on one warp (zero: M_ij starts from 0): lane (ti, tj) owns
// rows 8 ti .. +7 and columns 4 tj .. +3, so each quarter of the warp reads
// and writes 128 contiguous bytes.
__device__ __forceinline__ void panel_update(float* B, const float* Z, int ldz,
                                             int i0, int j0, bool zero) {
  const int lane = threadIdx.x & 31, ti = lane >> 3, tj = lane & 7;
  float4 acc[8];
  float4* row = reinterpret_cast<float4*>(B + 8 * ti * PLD + 4 * tj);
#pragma unroll
  for (int u = 0; u < 8; ++u)
    acc[u] = zero ? make_float4(0.f, 0.f, 0.f, 0.f) : row[u * (PLD / 4)];
  const float* zi = Z + i0 + 8 * ti;
  const float* zj = Z + j0 + 4 * tj;
#pragma unroll 4
  for (int k = 0; k < 32; ++k) {
    const float4 p = *reinterpret_cast<const float4*>(zi + k * ldz);
    const float4 q = *reinterpret_cast<const float4*>(zi + k * ldz + 4);
    const float4 b = *reinterpret_cast<const float4*>(zj + k * ldz);
    const float l[8] = {p.x, p.y, p.z, p.w, q.x, q.y, q.z, q.w};
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      acc[u].x -= l[u] * b.x;
      acc[u].y -= l[u] * b.y;
      acc[u].z -= l[u] * b.z;
      acc[u].w -= l[u] * b.w;
    }
  }
#pragma unroll
  for (int u = 0; u < 8; ++u) row[u * (PLD / 4)] = acc[u];
}

// The update of the next diagonal block, rows 8 h .. +7 on this warp (lane
// (ti, tj): two rows, four columns): the pivot chain waits for it, so four
// warps share it.
__device__ __forceinline__ void panel_update_quarter(float* B, const float* Zd,
                                                     int ldz, int h) {
  const int lane = threadIdx.x & 31, ti = lane >> 3, tj = lane & 7;
  const int r = 8 * h + 2 * ti;
  float4* row = reinterpret_cast<float4*>(B + r * PLD + 4 * tj);
  float4 a0 = row[0], a1 = row[PLD / 4];
#pragma unroll 8
  for (int k = 0; k < 32; ++k) {
    const float2 l = *reinterpret_cast<const float2*>(Zd + k * ldz + r);
    const float4 b = *reinterpret_cast<const float4*>(Zd + k * ldz + 4 * tj);
    a0.x -= l.x * b.x; a0.y -= l.x * b.y; a0.z -= l.x * b.z; a0.w -= l.x * b.w;
    a1.x -= l.y * b.x; a1.y -= l.y * b.y; a1.z -= l.y * b.z; a1.w -= l.y * b.w;
  }
  row[0] = a0;
  row[PLD / 4] = a1;
}

struct PanelOut {
  double* Linv = nullptr;  // may be null
  double* R = nullptr;     // FP64 L^{-T} (when split is null)
  float* split = nullptr;  // TF32 hi and lo of L^{-T}
  int ldm = 0;
  int split_diag = 0;      // leave the diagonal out, written as pairs
  // chol_refined: where any of nhopeless words is set, or max |Linv - I| is
  // 1/2 or more, *stop becomes 1 and Linv is of no use; else *stop is 0
  const int* hopeless = nullptr;
  int nhopeless = 0;
  unsigned long long* stop = nullptr;
};

template <bool dev>
__global__ void __launch_bounds__(kPanelThreads, 1)
    k_chol_panel(int m, const double* __restrict__ S,
                 const float* __restrict__ Bf, const float* __restrict__ Qf,
                 PanelOut out, IterScalars* sc,
                 const double* __restrict__ lpart, int nlpart) {
  extern __shared__ __align__(16) float psm[];
  __shared__ int bad;
  __shared__ float ydg[kPanelMax];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr int nw = kPanelThreads / 32;
  const int P = (m + 31) >> 5, mp = 32 * P, ldz = mp + 4;
  float* M = psm;
  float* Z = M + panel_blocks(P) * PSZ;
  float* lcol = Z + 32 * ldz;   // 32 x 32, and a line read past its end
  float* rd = lcol + 33 * 32;
  auto blk = [&](int i, int j) { return M + (panel_blocks(i) + j) * PSZ; };
  if (!dev && out.stop) {
    const bool any = tid < out.nhopeless && out.hopeless[tid];
    if (__syncthreads_or(any)) {
      if (tid == 0) *out.stop = 1ull;
      return;
    }
  }
  if (tid == 0) bad = 0;
  // S (or S(a) from B and Q) into the blocks, minus I in deviation form; the
  // padding is the identity. A unit is eight columns of a block, read along
  // its columns; with B and Q the mirrored unit is added after a barrier.
  const int units = 4 * panel_blocks(P);
  struct Unit {
    int bi, bj, g;
  };
  auto unit = [&](int u) {
    int bi = 0;
    while (panel_blocks(bi + 1) <= (u >> 2)) ++bi;
    return Unit{bi, (u >> 2) - panel_blocks(bi), 8 * (u & 3)};
  };
  auto load = [&](int u, bool mirror, float (&b)[8], float (&q)[8]) {
    const Unit t = unit(u);
    const int row = 32 * (mirror ? t.bj : t.bi) + lane;
    const int col = 32 * (mirror ? t.bi : t.bj) + t.g;
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const bool in = row < m && col + e < m;
      b[e] = in ? Bf[row + (col + e) * m] : 0.f;
      q[e] = in ? Qf[row + (col + e) * m] : 0.f;
    }
  };
  if (Bf) {
    // (the loads of three units are in flight while the line step is formed)
    constexpr int NU = 3;
    float b[NU][8], q[NU][8];
#pragma unroll
    for (int k = 0; k < NU; ++k)
      if (warp + k * nw < units) load(warp + k * nw, false, b[k], q[k]);
    float al, hq;
    if (lpart) {  // the line step (it sets sc->alpha)
      __shared__ double lq[4], la;
      if (warp < 4) {
        double v = lane < nlpart ? lpart[4 * (size_t)lane + warp] : 0.0;
        for (int k = lane + 32; k < nlpart; k += 32)
          v += lpart[4 * (size_t)k + warp];
        v = warp_sum(v);
        if (lane == 0) lq[warp] = v;
      }
      __syncthreads();
      if (tid == 0) la = line_alpha(m, lq, sc);
      __syncthreads();
      al = (float)la;
      hq = (float)(0.5 * la * la);
      if (tid == kPanelThreads - 1) line_store(lq, la, sc);
    } else {
      al = (float)sc->alpha;
      hq = (float)(0.5 * sc->alpha * sc->alpha);
    }
    for (int base = warp; base < units; base += NU * nw) {
#pragma unroll
      for (int k = 0; k < NU; ++k) {
        const int u = base + k * nw;
        if (u >= units) break;
        if (base != warp) load(u, false, b[k], q[k]);
        const Unit t = unit(u);
        const int row = 32 * t.bi + lane, col = 32 * t.bj + t.g;
        float v[8];
#pragma unroll
        for (int e = 0; e < 8; ++e)
          v[e] = al * b[k][e] + hq * q[k][e] +
                 (!dev && row == col + e ? 1.f : 0.f);
        float4* D =
            reinterpret_cast<float4*>(blk(t.bi, t.bj) + lane * PLD + t.g);
        D[0] = make_float4(v[0], v[1], v[2], v[3]);
        D[1] = make_float4(v[4], v[5], v[6], v[7]);
      }
    }
#pragma unroll
    for (int k = 0; k < NU; ++k)
      if (warp + k * nw < units) load(warp + k * nw, true, b[k], q[k]);
    __syncthreads();
    for (int base = warp; base < units; base += NU * nw) {
#pragma unroll
      for (int k = 0; k < NU; ++k) {
        const int u = base + k * nw;
        if (u >= units) break;
        if (base != warp) load(u, true, b[k], q[k]);
        const Unit t = unit(u);
        float* D = blk(t.bi, t.bj) + t.g * PLD + lane;
#pragma unroll
        for (int e = 0; e < 8; ++e) D[e * PLD] += al * b[k][e] + hq * q[k][e];
      }
    }
  } else {
    for (int u = warp; u < units; u += nw) {
      const Unit t = unit(u);
      const int row = 32 * t.bi + lane, col = 32 * t.bj + t.g;
      float* D = blk(t.bi, t.bj) + lane * PLD + t.g;
      double v[8];
#pragma unroll
      for (int e = 0; e < 8; ++e)
        v[e] = row < m && col + e < m
                   ? S[row + (col + e) * m] - (dev && row == col + e ? 1.0 : 0.0)
                   : (!dev && row == col + e ? 1.0 : 0.0);
#pragma unroll
      for (int e = 0; e < 8; ++e) D[e] = (float)v[e];
    }
  }
  __syncthreads();
  auto diag = [&](int p) {  // warps 0 and 1
    if (warp == 0) {
      float thr = 0.f;
      if (!dev) {
        // a pivot that has lost all but 4m roundings of its original diagonal
        // entry marks a (numerically) singular S
        const int c = 32 * p + lane;
        const double sjj = (Bf || c >= m) ? 1.0 : fabs(S[c + c * m]);
        thr = (float)(4 * m) * 1.2e-7f * (float)sjj;
      }
      const bool b = panel_factor<dev>(blk(p, p), thr, lcol, rd, ydg + 32 * p);
      if (lane == 0 && b) bad = 1;
    } else {
      panel_invert(blk(p, p), lcol, rd);
    }
  };
  if (warp < 2) diag(0);
  __syncthreads();
  for (int p = 0; p < P && P > 1; ++p) {
    // (2) the panel Z: warp units are (block column, half of the 32 rows)
    const float* X = blk(p, p);
    const int xq = lane & 7;
    for (int u = warp; u < 2 * P; u += nw) {
      const int b = u >> 1, k0 = 16 * (u & 1) + 4 * (lane >> 3);
      float acc[4][4] = {};
      const int kend = 16 * (u & 1) + 16;  // X_pp is lower triangular
      if (b > p) {  // L_bp(x, k) = sum_q A_bp(x, q) X_pp(k, q), x = xq + 8 v
        const float* A = blk(b, p);
        for (int q = 0; q < kend; q += 4) {
          float4 a[4], x[4];
#pragma unroll
          for (int v = 0; v < 4; ++v) {
            a[v] = *reinterpret_cast<const float4*>(A + (xq + 8 * v) * PLD + q);
            x[v] = *reinterpret_cast<const float4*>(X + (k0 + v) * PLD + q);
          }
#pragma unroll
          for (int s = 0; s < 4; ++s)
#pragma unroll
            for (int v = 0; v < 4; ++v)
              acc[s][v] += x[s].x * a[v].x + x[s].y * a[v].y +
                           x[s].z * a[v].z + x[s].w * a[v].w;
        }
#pragma unroll
        for (int s = 0; s < 4; ++s)
#pragma unroll
          for (int v = 0; v < 4; ++v)
            Z[(k0 + s) * ldz + 32 * b + xq + 8 * v] = acc[s][v];
      } else if (b < p) {  // X_pb(k, x) = sum_q X_pp(k, q) W_pb(q, x)
        const float* W = blk(p, b);
        for (int q = 0; q < kend; q += 4) {
          float4 x[4];
#pragma unroll
          for (int s = 0; s < 4; ++s)
            x[s] = *reinterpret_cast<const float4*>(X + (k0 + s) * PLD + q);
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const float4 t =
                *reinterpret_cast<const float4*>(W + (q + e) * PLD + 4 * xq);
#pragma unroll
            for (int s = 0; s < 4; ++s) {
              const float xe = e == 0 ? x[s].x : e == 1 ? x[s].y
                             : e == 2 ? x[s].z : x[s].w;
              acc[s][0] += xe * t.x;
              acc[s][1] += xe * t.y;
              acc[s][2] += xe * t.z;
              acc[s][3] += xe * t.w;
            }
          }
        }
#pragma unroll
        for (int s = 0; s < 4; ++s)
          *reinterpret_cast<float4*>(Z + (k0 + s) * ldz + 32 * b + 4 * xq) =
              make_float4(acc[s][0], acc[s][1], acc[s][2], acc[s][3]);
      } else {
#pragma unroll
        for (int s = 0; s < 4; ++s)
          *reinterpret_cast<float4*>(Z + (k0 + s) * ldz + 32 * b + 4 * xq) =
              *reinterpret_cast<const float4*>(X + (k0 + s) * PLD + 4 * xq);
      }
    }
    __syncthreads();
    // (3) block updates; row p takes its final values X_pj from Z
    const int nupd = panel_blocks(P) - panel_blocks(p + 1);
    const bool more = p + 1 < P;
    if (more && warp < 4) {
      panel_update_quarter(blk(p + 1, p + 1), Z + 32 * (p + 1), ldz, warp);
      asm volatile("bar.sync 9, 128;" ::: "memory");
    }
    if (more && warp < 2) {
      diag(p + 1);
    } else {
      const int w0 = more ? warp - 2 : warp, wn = more ? nw - 2 : nw;
      for (int u = w0; u < nupd + p; u += wn) {
        if (u < nupd) {
          const int b = panel_blocks(p + 1) + u;
          int bi = p + 1;
          while (panel_blocks(bi + 1) <= b) ++bi;
          const int bj = b - panel_blocks(bi);
          if (bi == p + 1 && bj == p + 1) continue;  // done above
          panel_update(blk(bi, bj), Z, ldz, 32 * bi, 32 * bj, bj == p);
        } else {
          const int bj = u - nupd;
          float* D = blk(p, bj);
#pragma unroll
          for (int k = 0; k < 32; k += 4) {
            const int r = k + (lane >> 3);
            *reinterpret_cast<float4*>(D + r * PLD + 4 * xq) =
                *reinterpret_cast<const float4*>(Z + r * ldz + 32 * bj + 4 * xq);
          }
        }
      }
    }
    __syncthreads();
  }
  const bool isbad = bad != 0;
  // column i of R = L^{-T} is row i of X: contiguous in its block row
  auto entry = [&](int k, int i) -> float {  // off the diagonal, k < i
    return isbad ? 0.f : blk(i >> 5, k >> 5)[(i & 31) * PLD + (k & 31)];
  };
  auto dfull = [&](int i) -> float {  // deviation form: y_ii, else x_ii
    return isbad ? (dev ? 0.f : 1.f)
                 : (dev ? ydg[i] : blk(i >> 5, i >> 5)[(i & 31) * (PLD + 1)]);
  };
  if (out.split) {
    float* hi = out.split;
    float* lo = hi + (size_t)out.ldm * m;
    float* dg = lo + (size_t)out.ldm * m;
    // Four entries of a column per lane at a time. Only the triangle: the zeros
    // below it stay from the buffer's allocation (one SM's stores, not the
    // arithmetic, are what this phase takes).
    for (int i = warp; i < m; i += nw) {
      const float* X = blk(i >> 5, 0) + (i & 31) * PLD + lane;
      float* ph = hi + (size_t)i * out.ldm;
      float* pl = lo + (size_t)i * out.ldm;
      for (int k0 = 0; k0 < i; k0 += 128) {
        float x[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const int k = k0 + 32 * e + lane;
          x[e] = k < i && !isbad ? X[((k0 >> 5) + e) * PSZ] : 0.f;
        }
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const int k = k0 + 32 * e + lane;
          if (k < i) {
            const float h = tc::tf32_rna(x[e]);
            ph[k] = h;
            pl[k] = tc::tf32_rna(x[e] - h);
          }
        }
      }
    }
    for (int i = tid; i < m; i += kPanelThreads) {  // the diagonal
      const float y = dfull(i);
      float h = 0.f, l = 0.f;
      if (out.split_diag) {
        const F2 d = dev ? two_sum(1.f, y) : F2{y, 0.f};
        dg[i] = d.h;
        dg[m + i] = d.l;
      } else if (dev) {
        h = tc::tf32_rna(1.f + y);
        l = tc::tf32_rna(y - (h - 1.f));
      } else {
        h = tc::tf32_rna(y);
        l = tc::tf32_rna(y - h);
      }
      hi[i + (size_t)i * out.ldm] = h;
      lo[i + (size_t)i * out.ldm] = l;
    }
  } else if (out.R) {
    for (int i = warp; i < m; i += nw)
      for (int k = lane; k < m; k += 32)
        out.R[k + i * m] = k < i ? to_f64(entry(k, i))
                         : k > i ? 0.0
                                 : (dev ? 1.0 : 0.0) + (double)dfull(i);
  }
  float far = 0.f;  // max |Linv - I|
  if (out.Linv)
    for (int k = warp; k < m; k += nw)
      for (int i = lane; i < m; i += 32) {
        const float x = i > k ? entry(k, i) : i == k ? dfull(i) : 0.f;
        far = fmaxf(far, fabsf(!dev && i == k ? x - 1.f : x));
        out.Linv[i + k * m] =
            i == k ? (dev ? 1.0 : 0.0) + (double)x : to_f64(x);
      }
  if (!dev && out.stop) {
    const bool in_vain = __syncthreads_or(isbad || !(far < 0.5f));
    if (tid == 0) *out.stop = in_vain ? 1ull : 0ull;
  }
  if (tid == 0 && isbad && sc) sc->status |= 1;
}

// ---------------------------------------------------------------------------
// Blocked Cholesky S = L L^T and L^{-1} on many CTAs, for large m (Fig. ONFIG
// steps (2), (3)): the same arithmetic as k_chol_inv, spread over launches.
// The padded working copy W (mp x mp, leading dimension mp, lower triangle)
// is factorised right-looking over 32-column panels: per panel p, one CTA
// factors the diagonal block and inverts it (k_cb_diag); then every lower
// tile (I, J) of the trailing matrix, on its own CTA, solves its two panel
// blocks against the diagonal block's inverse, L_Ip = A_Ip X_pp^T, and
// subtracts L_Ip L_Jp^T (k_cb_update); the diagonal tile's CTA stores L_Ip.
// L^{-1} = X follows by recursive doubling: for a diagonal block split as
// [A 0; B C], its inverse is [A^{-1} 0; -C^{-1} B A^{-1}  C^{-1}], so with the
// 32 x 32 inverses from k_cb_diag, levels of block size 32, 64, ... each form
// T = B A^{-1}, then X_CA = -C^{-1} T, for all blocks of the level at once
// (k_cb_inv). Deviation form (dev): W holds S - I, L = I + F
// and X = I + Y with the identities implicit, so FP32 arithmetic keeps L to
// FP64 accuracy relative to I when S is close to I.
// ---------------------------------------------------------------------------
constexpr int CB = 32;

// A power of two whose square brings a positive number into [1/2, 2) (finite
// for any bits); 1 for a number on either side of 1
__device__ __forceinline__ double half_exp_scale(double x) {
  const int e = (int)((__double_as_longlong(x) >> 52) & 0x7ff) - 1023;
  return __longlong_as_double((long long)(1023 - ((e + 1) >> 1)) << 52);
}

// S' = D S D (D from S's diagonal; the lower triangle of S, mirrored), or S(a)
// = I + a (B + B^T) + a^2 (Q + Q^T) / 2. Clears the deviations. hopeless[CTA]:
// does it hold two columns with a cosine above 1/2? Their own entry of L^{-1}
// (c / sqrt(1 - c^2) for unit columns) is then about what refined_ok refuses,
// and the attempt ends here.
__global__ void __launch_bounds__(256)
    k_ref_form(int m, const double* __restrict__ S,
               const double* __restrict__ Bm, const double* __restrict__ Q,
               const IterScalars* __restrict__ sc, double* __restrict__ Sp,
               unsigned long long* dev, int* hopeless) {
  const int e = blockIdx.x * 256 + threadIdx.x;
  if (e < kRefStop) dev[e] = 0ull;
  bool far = false;
  if (e < m * m) {
    const int i = max(e % m, e / m), k = min(e % m, e / m);
    double v;
    if (Bm) {
      const double al = sc->alpha;
      v = al * (Bm[i + k * m] + Bm[k + i * m]) +
          0.5 * al * al * (Q[i + k * m] + Q[k + i * m]) + (i == k ? 1.0 : 0.0);
    } else {
      const double sii = S[i + i * m], skk = S[k + k * m];
      const double di = half_exp_scale(sii), dk = half_exp_scale(skk);
      v = S[i + k * m] * di * dk;
      far = i != k && 4.0 * v * v > (sii * di * di) * (skk * dk * dk);
    }
    Sp[e] = v;
  }
  const int any = __syncthreads_or(far);
  if (threadIdx.x == 0) hopeless[blockIdx.x] = any;
}

// L^{-1} = X D and its transpose, where the corrections converged
__global__ void __launch_bounds__(256)
    k_ref_out(int m, const double* __restrict__ S, const double* __restrict__ X,
              const unsigned long long* __restrict__ dev,
              double* __restrict__ Linv, double* __restrict__ R) {
  if (!refined_ok(dev)) return;
  const int e = blockIdx.x * 256 + threadIdx.x;
  if (e >= m * m) return;
  const int i = e % m, k = e / m;
  const double lo = i >= k ? X[e] * (S ? half_exp_scale(S[k + k * m]) : 1.0) : 0.0;
  const double up = i <= k ? X[k + i * m] * (S ? half_exp_scale(S[i + i * m]) : 1.0)
                           : 0.0;
  if (Linv) Linv[e] = lo;
  R[e] = up;
}

// The line step alpha from the line-term partials (one CTA).
__global__ void k_cb_alpha(int m, const double* __restrict__ lpart, int nlpart,
                           IterScalars* sc) {
  __shared__ double lred[4 * 32];
  line_alpha_block(m, lpart, nlpart, sc, lred);
}

// W <- lower triangle of S, or of S(a) = I + a (B + B^T) + a^2 Q (Q
// symmetric), minus I in deviation form; the padding is the identity (zero
// in deviation form). Clears the failure flag.
template <typename Tm, bool dev>
__global__ void k_cb_form(int m, int mp, const double* __restrict__ S,
                          const double* __restrict__ Bm,
                          const double* __restrict__ Q,
                          const float* __restrict__ Bf,
                          const float* __restrict__ Qf,
                          const IterScalars* __restrict__ sc, Tm* __restrict__ W,
                          int* bad) {
  const int64_t total = (int64_t)mp * mp;
  if (blockIdx.x == 0 && threadIdx.x == 0) *bad = 0;
  const double al = (Bm || Bf) ? sc->alpha : 0.0;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int i = (int)(e % mp), k = (int)(e / mp);
    if (i < k) continue;  // the upper triangle is never read
    double v;
    if (i < m && k < m) {
      // a (B + B^T) + a^2 (Q + Q^T) / 2, as k_chol_inv forms it
      if (Bf)
        v = (double)((float)al * (Bf[i + k * m] + Bf[k + i * m]) +
                     (float)(0.5 * al * al) * (Qf[i + k * m] + Qf[k + i * m]));
      else if (Bm)
        v = al * (Bm[i + (int64_t)k * m] + Bm[k + (int64_t)i * m]) +
            0.5 * al * al * (Q[i + (int64_t)k * m] + Q[k + (int64_t)i * m]);
      else
        v = S[i + (int64_t)k * m] - (dev && i == k ? 1.0 : 0.0);
      if ((Bm || Bf) && !dev && i == k) v += 1.0;
    } else {
      v = (!dev && i == k) ? 1.0 : 0.0;
    }
    W[e] = (Tm)v;
  }
}

// Factor and invert the 32 x 32 diagonal block of panel p: warp 0 runs
// diag_factor_warp and diag_inverse_warp; all 256 threads write the inverse.
// Writes the block of L (F in deviation form; zeros above the diagonal) and
// of X = L^{-1} (Y in deviation form).
template <typename Tm, bool dev>
__global__ void __launch_bounds__(256, 1)
    k_cb_diag(int m, int mp, int p, const double* __restrict__ S,
              bool from_S, const Tm* __restrict__ W, Tm* __restrict__ L,
              Tm* __restrict__ X, int* bad) {
  __shared__ Tm B[32 * 33];  // the block, column-major, leading dimension 33
  __shared__ Tm rd[32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int c0 = CB * p, r = c0 + lane;
  const Tm eps = sizeof(Tm) == 4 ? (Tm)1.2e-7 : (Tm)2.3e-16;
  if (warp == 0) {
    Tm w[32];
#pragma unroll
    for (int j = 0; j < 32; ++j) w[j] = W[r + (size_t)(c0 + j) * mp];
    Tm thr = (Tm)0;
    if (!dev) {
      const double sjj = (!from_S || r >= m) ? 1.0 : fabs(S[r + (int64_t)r * m]);
      thr = (Tm)(4 * m) * eps * (Tm)sjj;
    }
    const bool b = diag_factor_warp<Tm, dev>(w, thr, rd);
    // the block of L (lower, zeros above) to global and to shared memory
#pragma unroll
    for (int j = 0; j < 32; ++j) {
      const Tm x = lane >= j ? w[j] : (Tm)0;
      L[r + (size_t)(c0 + j) * mp] = x;
      B[lane + 33 * j] = x;
    }
    if (lane == 0 && b) atomicOr(bad, 1);
    __syncwarp();
    Tm x[32];
    diag_inverse_warp<Tm, dev>(B, 33, rd, x);
    __syncwarp();  // every lane has read L before the block is replaced
#pragma unroll
    for (int i = 0; i < 32; ++i) B[i + 33 * lane] = x[i];
  }
  __syncthreads();
  for (int e = tid; e < 32 * 32; e += 256) {
    const int i = e & 31, j = e >> 5;
    X[(c0 + i) + (size_t)(c0 + j) * mp] = i >= j ? B[i + 33 * j] : (Tm)0;
  }
}

// Trailing update of panel p: CTA t takes the lower tile (I, J), p < J <= I,
// of the trailing matrix. L_I = A_I X_pp^T (deviation form: A_I + A_I Y_pp^T)
// for the panel blocks of rows I and J, then W_IJ -= L_I L_J^T; the CTA of
// the diagonal tile writes L_I into L.
template <typename Tm, bool dev>
__global__ void __launch_bounds__(256)
    k_cb_update(int mp, int p, Tm* __restrict__ W, Tm* __restrict__ L,
                const Tm* __restrict__ X) {
  __shared__ Tm Xp[32][33], AI[32][33], AJ[32][33], LI[32][33], LJ[32][33];
  const int tid = threadIdx.x;
  const int P = mp / CB;
  // tile t -> (I, J), J <= I, counted over rows I = p + 1 .. P - 1
  const int t = blockIdx.x;
  int a = (int)((sqrtf(8.0f * t + 1.0f) - 1.0f) * 0.5f);
  while ((a + 1) * (a + 2) / 2 <= t) ++a;
  while (a * (a + 1) / 2 > t) --a;
  const int I = p + 1 + a, J = p + 1 + (t - a * (a + 1) / 2);
  if (I >= P) return;
  const int c0 = CB * p, i0 = CB * I, j0 = CB * J;
  for (int e = tid; e < 32 * 32; e += 256) {
    const int i = e & 31, k = e >> 5;
    Xp[i][k] = X[(c0 + i) + (size_t)(c0 + k) * mp];
    AI[i][k] = W[(i0 + i) + (size_t)(c0 + k) * mp];
    AJ[i][k] = W[(j0 + i) + (size_t)(c0 + k) * mp];
  }
  __syncthreads();
  const int r = tid & 31, cb = (tid >> 5) * 4;
  // L_I (and L_J) rows: L[r][c] = sum_{k <= c} A[r][k] X[c][k] (+ A[r][c])
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int c = cb + u;
    Tm sI = dev ? AI[r][c] : (Tm)0, sJ = dev ? AJ[r][c] : (Tm)0;
    for (int k = 0; k <= c; ++k) {
      sI += AI[r][k] * Xp[c][k];
      sJ += AJ[r][k] * Xp[c][k];
    }
    LI[r][c] = sI;
    LJ[r][c] = sJ;
  }
  __syncthreads();
  if (I == J)
    for (int e = tid; e < 32 * 32; e += 256) {
      const int i = e & 31, k = e >> 5;
      L[(i0 + i) + (size_t)(c0 + k) * mp] = LI[i][k];
    }
  // W_IJ -= L_I L_J^T: thread (r, cb..cb+3)
  Tm acc[4] = {0, 0, 0, 0};
#pragma unroll 8
  for (int k = 0; k < 32; ++k) {
    const Tm li = LI[r][k];
#pragma unroll
    for (int u = 0; u < 4; ++u) acc[u] += li * LJ[cb + u][k];
  }
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const size_t o = (i0 + r) + (size_t)(j0 + cb + u) * mp;
    W[o] -= acc[u];
  }
}

// One level of the recursive inverse, block size s: pair q has A = rows and
// columns [2 q s, 2 q s + s) and C = [2 q s + s, 2 q s + 2 s) (cut at mp);
// phase 0: T_CA = L_CA X_A (deviation form: F_CA + F_CA Y_A), phase 1:
// X_CA = -X_C T_CA (deviation form: -(T + Y_C T)). One CTA per 32 x 32 tile
// of C x A (blockIdx.y), pairs along blockIdx.x.
template <typename Tm, bool dev>
__global__ void __launch_bounds__(256)
    k_cb_inv(int mp, int s, int phase, const Tm* __restrict__ L,
             Tm* __restrict__ X, Tm* __restrict__ T) {
  __shared__ Tm Ls[32][33], Rs[32][33];
  const int tid = threadIdx.x;
  const int a0 = 2 * s * blockIdx.x, c0 = a0 + s;
  if (c0 >= mp) return;
  const int nc = min(s, mp - c0);           // rows of C (multiple of 32)
  const int tiles_a = s / CB;
  const int ti = blockIdx.y / tiles_a, tj = blockIdx.y % tiles_a;
  if (CB * ti >= nc) return;
  const int gi = c0 + CB * ti, gj = a0 + CB * tj;  // output tile origin
  const int r = tid & 31, cb = (tid >> 5) * 4;
  Tm acc[4] = {0, 0, 0, 0};
  // phase 0: sum over k in A of L[gi.., k] X[k, gj..] (X_A lower: k >= gj)
  // phase 1: sum over k in C of X[gi.., k] T[k, gj..] (X_C lower: k <= gi+31)
  const int kb = phase == 0 ? gj : c0;
  const int ke = phase == 0 ? a0 + s : gi + CB;
  for (int k0 = kb; k0 < ke; k0 += CB) {
    for (int e = tid; e < 32 * 32; e += 256) {
      const int i = e & 31, k = e >> 5;
      if (phase == 0) {
        Ls[i][k] = L[(gi + i) + (size_t)(k0 + k) * mp];
        Rs[k][i] = X[(k0 + k) + (size_t)(gj + i) * mp];   // Rs[k][col]
      } else {
        Ls[i][k] = X[(gi + i) + (size_t)(k0 + k) * mp];
        Rs[k][i] = T[(k0 + k) + (size_t)(gj + i) * mp];
      }
    }
    __syncthreads();
#pragma unroll 8
    for (int k = 0; k < 32; ++k) {
      const Tm l = Ls[r][k];
#pragma unroll
      for (int u = 0; u < 4; ++u) acc[u] += l * Rs[k][cb + u];
    }
    __syncthreads();
  }
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const size_t o = (gi + r) + (size_t)(gj + cb + u) * mp;
    if (phase == 0)
      T[o] = acc[u] + (dev ? L[o] : (Tm)0);
    else
      X[o] = -(acc[u] + (dev ? T[o] : (Tm)0));
  }
}

// R = L^{-T} (upper) and Linv = L^{-1} (lower) in FP64 from X; identities
// and status bit 1 when a pivot failed.
template <typename Tm, bool dev>
__global__ void k_cb_out(int m, int mp, const Tm* __restrict__ X,
                         double* __restrict__ Linv, double* __restrict__ R,
                         const int* bad, IterScalars* sc) {
  const int isbad = *bad;
  const int64_t total = (int64_t)m * m;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int i = (int)(e % m), k = (int)(e / m);  // Linv(i, k) = R(k, i)
    double v = 0.0;
    if (isbad) {
      if (i == k) v = 1.0;
    } else if (i >= k) {
      v = (double)X[i + (size_t)k * mp];
      if (dev && i == k) v += 1.0;
    }
    if (Linv) Linv[e] = v;
    R[k + (int64_t)i * m] = v;
  }
  if (blockIdx.x == 0 && threadIdx.x == 0 && isbad && sc) sc->status |= 1;
}

// ---------------------------------------------------------------------------
// Line-model terms over 32 x 32 tiles of the (i, j) index space, one CTA of
// 1024 threads per tile, partial sums to part[tile * 4 + q]:
//   q = 0: tr(D1) = -tr(W)
//   q = 1: tr(D2) = tr(P^T H P) - sum_ij Q_ij A0_ij
//   q = 2: tr(S1 D1) = sum_ij A0_ij (B B^T - B^T B)_ij
//                      - 1/2 sum_ij S1_ij (W_ij + W_ji)
//   q = 3: tr(Q)
// with A0 = sym(H') + diag(H_D), S1 = B + B^T; tr(S1 (A0 B - B A0)) reduces
// to tr(A0 (B B^T - B^T B)) by cyclic invariance, so no m x m product is
// stored.
// ---------------------------------------------------------------------------
template <typename Tm>
__global__ void __launch_bounds__(1024)
    k_line_terms(int m, const Tm* __restrict__ Hp,
                 const double* __restrict__ HD, const Tm* __restrict__ Bm,
                 const Tm* __restrict__ Q, const double* __restrict__ hpd,
                 int hpd_stride, const double* __restrict__ tr_parts,
                 int n_tr_parts, const Tm* __restrict__ W,
                 double* __restrict__ part) {
  __shared__ Tm t0[32][33], t1[32][33], t2[32][33], t3[32][33];
  __shared__ double red[4 * 32];
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const int I0 = blockIdx.x * 32, J0 = blockIdx.y * 32;
  const int i = I0 + tx, j = J0 + ty;
  // blockIdx.z splits the k range of M = B B^T - B^T B; every other term is
  // added by the first split only (the sums are linear in M)
  const int ks = blockIdx.z, KS = gridDim.z;
  Tm M = 0;
  for (int k0 = 32 * ks; k0 < m; k0 += 32 * KS) {
    t0[tx][ty] = (I0 + tx < m && k0 + ty < m) ? (Tm)Bm[(I0 + tx) + (k0 + ty) * m] : (Tm)0;
    t1[tx][ty] = (J0 + tx < m && k0 + ty < m) ? (Tm)Bm[(J0 + tx) + (k0 + ty) * m] : (Tm)0;
    t2[tx][ty] = (k0 + tx < m && I0 + ty < m) ? (Tm)Bm[(k0 + tx) + (I0 + ty) * m] : (Tm)0;
    t3[tx][ty] = (k0 + tx < m && J0 + ty < m) ? (Tm)Bm[(k0 + tx) + (J0 + ty) * m] : (Tm)0;
    __syncthreads();
#pragma unroll 8
    for (int kk = 0; kk < 32; ++kk)
      M += t0[tx][kk] * t1[ty][kk] - t2[kk][tx] * t3[kk][ty];
    __syncthreads();
  }
  // transposed tiles (J, I) of H', B, W for the (j, i) entries
  t0[tx][ty] = (J0 + tx < m && I0 + ty < m) ? (Tm)Hp[(J0 + tx) + (I0 + ty) * m] : (Tm)0;
  t1[tx][ty] = (J0 + tx < m && I0 + ty < m) ? (Tm)Bm[(J0 + tx) + (I0 + ty) * m] : (Tm)0;
  t2[tx][ty] = (J0 + tx < m && I0 + ty < m) ? (Tm)W[(J0 + tx) + (I0 + ty) * m] : (Tm)0;
  __syncthreads();
  Tm v0 = 0, v1 = 0, v2 = 0, v3 = 0;
  if (i < m && j < m) {
    const int e = i + j * m;
    const Tm a0 = (Tm)0.5 * ((Tm)Hp[e] + t0[ty][tx]) + (i == j ? (Tm)HD[i] : (Tm)0);
    v2 = a0 * M;
    if (ks == 0) {
      const Tm bij = (Tm)Bm[e], qij = (Tm)Q[e];
      const Tm s1 = bij + t1[ty][tx];
      const Tm wij = (Tm)W[e], wji = t2[ty][tx];
      v2 -= (Tm)0.5 * s1 * (wij + wji);
      v1 = -qij * a0;
      if (i == j) {
        v0 = -wij;
        if (hpd) v1 += (Tm)hpd[(size_t)i * hpd_stride];
        v3 = (Tm)Q[e];
      }
    }
  }
  // the sums over the CTA: FP64, or for FP32 terms double-float pairs within
  // each warp (an FP64 add of every thread would take most of the kernel)
  double v[4];
  const int cta = blockIdx.y * gridDim.x + blockIdx.x;
  const int ncta = gridDim.x * gridDim.y;
  if constexpr (sizeof(Tm) == 4) {
    F2 p[4] = {{v0, 0.f}, {v1, 0.f}, {v2, 0.f}, {v3, 0.f}};
    if (tr_parts && ks == 0)
      // tr(P^T H P) as the sum of the stencil's partial column dots, each
      // first-split CTA adding a fixed share
      for (int k = cta * blockDim.x + threadIdx.x; k < n_tr_parts;
           k += ncta * blockDim.x)
        p[1] = df_add(p[1], df_of_bits(tr_parts[k]));
    const F2 t = warp_sum4(
        p,
        [](F2 x, int o) {
          return F2{__shfl_xor_sync(0xffffffffu, x.h, o),
                    __shfl_xor_sync(0xffffffffu, x.l, o)};
        },
        [](F2 x, F2 y) { return df_add(x, y); });
    if ((tx & 7) == 0) red[(tx >> 3) * 32 + ty] = to_f64(t.h) + to_f64(t.l);
    block_sum4_finish(v, red, blockDim.x >> 5);
  } else {
    v[0] = v0;
    v[1] = v1;
    v[2] = v2;
    v[3] = v3;
    if (tr_parts && ks == 0)
      for (int k = cta * blockDim.x + threadIdx.x; k < n_tr_parts;
           k += ncta * blockDim.x)
        v[1] += tr_parts[k];
    block_sum4(v, red);
  }
  if (threadIdx.x == 0) {
    const size_t b =
        ((size_t)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
#pragma unroll
    for (int q = 0; q < 4; ++q) part[b * 4 + q] = v[q];
  }
}

// ---------------------------------------------------------------------------
// Cyclic Jacobi with the round-robin ordering: in each round m/2 disjoint
// (p, q) pairs are annihilated at once (columns, then rows, then Z). One CTA;
// A lives in shared memory (leading dimension m + 1) when it fits, else in
// the global work copy; Z accumulates in global memory, where its column
// updates are contiguous. T is the arithmetic type. Z starts from Z0 (FP64,
// may be null for the identity), so Z = Z0 J. A rotation is skipped when
// |a_pq| <= rot_tol (|a_pp| + |a_qq|) + abs_c ||A||_F (the second term sits
// above the rounding noise of the arithmetic type, so the sweeps end); they
// stop when one applied no rotation or the off-diagonal part is below
// conv_tol of the whole (squared Frobenius norms).
// ---------------------------------------------------------------------------
//
// Before a sweep all pairs are looked at together: when none would be rotated,
// its rounds are not run (m = 64 in FP64: 110 us of rounds).
template <typename T>
__global__ void __launch_bounds__(1024)
    k_jacobi(int m, const double* __restrict__ Ain, T* __restrict__ Ag,
             T* __restrict__ Zw, const double* __restrict__ Z0,
             double* __restrict__ w, double* __restrict__ Z, int* info,
             int max_sweeps, T rot_tol, T abs_c, T conv_tol, int use_smem) {
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ T cs[512], sn[512];
  __shared__ int pp[512], qq[512];
  __shared__ double red[2 * 32];
  __shared__ int done, rotated;
  __shared__ T abs_tol;
  const int tid = threadIdx.x, nt = blockDim.x;
  const int lane = tid & 31, warp = tid >> 5, nw = nt >> 5;
  const int ld = use_smem ? m + 1 : m;
  T* A = use_smem ? reinterpret_cast<T*>(smraw) : Ag;
  for (int c = warp; c < m; c += nw)
    for (int r = lane; r < m; r += 32) A[r + c * ld] = (T)Ain[r + c * m];
  for (int c = warp; c < m; c += nw)
    for (int r = lane; r < m; r += 32)
      Zw[r + c * m] = Z0 ? (T)Z0[r + c * m] : (r == c ? (T)1 : (T)0);
  const int M = m + (m & 1);
  const int np = M / 2;
  int sweeps = 0;
  bool settled = false;
  if (tid == 0) rotated = 1;
  __syncthreads();
  for (int sweep = 0; sweep <= max_sweeps; ++sweep) {
    double v[2] = {0.0, 0.0};
    for (int c = warp; c < m; c += nw)
      for (int r = lane; r < m; r += 32) {
        const double x = (double)A[r + c * ld];
        if (r == c)
          v[1] += x * x;
        else
          v[0] += x * x;
      }
    block_sum<2>(v, red);
    if (tid == 0) {
      done = (v[0] <= (double)conv_tol * (v[0] + v[1])) || !rotated ||
             sweep == max_sweeps;
      if (sweep == 0) abs_tol = (T)((double)abs_c * sqrt(v[0] + v[1]));
      rotated = 0;  // before the barrier: the rounds below may set it
    }
    __syncthreads();
    if (done) break;
    int any = 0;
    for (int c = warp; c < m; c += nw)
      for (int r = lane; r < c; r += 32) {
        const T x = A[r + c * ld];
        any |= x != (T)0 &&
               fabs(x) > rot_tol * (fabs(A[r + r * ld]) + fabs(A[c + c * ld])) +
                             abs_tol;
      }
    settled = !__syncthreads_or(any);
    sweeps = sweep + 1;
    if (settled) break;
    for (int r = 0; r < M - 1; ++r) {
      for (int k = tid; k < np; k += nt) {
        const int a0 = (k == 0) ? 0 : 1 + ((k - 1 + r) % (M - 1));
        const int kb = M - 1 - k;
        const int b0 = 1 + ((kb - 1 + r) % (M - 1));
        const int p = min(a0, b0), q = max(a0, b0);
        T c = 1, s = 0;
        if (q < m) {
          const T apq = A[p + q * ld];
          const T app = A[p + p * ld];
          const T aqq = A[q + q * ld];
          if (apq != (T)0 &&
              fabs(apq) > rot_tol * (fabs(app) + fabs(aqq)) + abs_tol) {
            const T th = (aqq - app) / ((T)2 * apq);
            T t;
            if (fabs(th) > (T)1e18)
              t = (T)0.5 / th;
            else
              t = (th >= (T)0 ? (T)1 : (T)-1) / (fabs(th) + sqrt(th * th + (T)1));
            c = (T)1 / sqrt(t * t + (T)1);
            s = t * c;
            rotated = 1;
          }
        }
        cs[k] = c;
        sn[k] = s;
        pp[k] = p;
        qq[k] = min(q, m - 1);
      }
      __syncthreads();
      for (int k = warp; k < np; k += nw) {  // A <- A J (columns p, q)
        const T s = sn[k];
        if (s == (T)0) continue;
        const T c = cs[k];
        T* ap = A + pp[k] * ld;
        T* aq = A + qq[k] * ld;
        for (int i0 = lane; i0 < m; i0 += 128) {
          T x[4], y[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int i = i0 + 32 * u;
            x[u] = i < m ? ap[i] : (T)0;
            y[u] = i < m ? aq[i] : (T)0;
          }
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int i = i0 + 32 * u;
            if (i < m) {
              ap[i] = c * x[u] - s * y[u];
              aq[i] = s * x[u] + c * y[u];
            }
          }
        }
      }
      __syncthreads();
      for (int k = warp; k < np; k += nw) {  // A <- J^T A (rows), Z <- Z J
        const T s = sn[k];
        if (s == (T)0) continue;
        const T c = cs[k];
        const int p = pp[k], q = qq[k];
        T* zp = Zw + p * m;
        T* zq = Zw + q * m;
        for (int j0 = lane; j0 < m; j0 += 128) {
          T x[4], y[4], u_[4], t_[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int jc = j0 + 32 * u;
            x[u] = jc < m ? A[p + jc * ld] : (T)0;
            y[u] = jc < m ? A[q + jc * ld] : (T)0;
            u_[u] = jc < m ? zp[jc] : (T)0;
            t_[u] = jc < m ? zq[jc] : (T)0;
          }
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const int jc = j0 + 32 * u;
            if (jc < m) {
              A[p + jc * ld] = c * x[u] - s * y[u];
              A[q + jc * ld] = s * x[u] + c * y[u];
              zp[jc] = c * u_[u] - s * t_[u];
              zq[jc] = s * u_[u] + c * t_[u];
            }
          }
        }
      }
      __syncthreads();
    }
  }
  // ascending order (stable on ties), a column per warp
  __syncthreads();
  for (int i = warp; i < m; i += nw) {
    const T wi = A[i + i * ld];
    int rank = 0;
    for (int j = lane; j < m; j += 32) {
      const T wj = A[j + j * ld];
      rank += (wj < wi) || (wj == wi && j < i);
    }
    rank = __reduce_add_sync(0xffffffffu, rank);
    if (lane == 0) w[rank] = (double)wi;
    for (int r = lane; r < m; r += 32) Z[r + rank * m] = (double)Zw[r + i * m];
  }
  if (tid == 0 && info) *info = (done || settled) ? sweeps : -1;
}

// ---------------------------------------------------------------------------
// One correction of an approximate eigenvector matrix X of a symmetric A, by
// the refinement of Ogita and Aishima (2018), derived to first order from
// (I + E)^T (X^T X) (I + E) = I and (I + E)^T (X^T A X) (I + E) diagonal:
// with R = I - X^T X and S = X^T A X,
//   lambda_i = s_ii / (1 - r_ii),
//   e_ij = (s_ij + lambda_j r_ij) / (lambda_j - lambda_i)  if the two are
//          further apart than delta = 2 (||S - diag(lambda)|| + ||A|| ||R||),
//   e_ij = r_ij / 2 otherwise, and also where the first-order step would
//          exceed 0.01 (inside a cluster only orthonormality is restored;
//          the closing FP64 Jacobi separates the cluster),
// and X <- X + X E. The 2-norms in delta are taken as 2 / sqrt(m) of the
// Frobenius norms, as for a matrix of random entries (m >= 128; the factor of
// m = 128 below that: a delta as large as the Frobenius norms leaves pairs of
// close eigenvalues to the FP64 sweeps, 170 us of them at m = 64, and with
// couplings up to their threshold), max |lambda_i| as ||A||. G = X^T X,
// S = X^T A X in, E out.
// ---------------------------------------------------------------------------
// Partial sums of ||S - D||^2 and ||R||^2 (R = I - G, D = diag(s_ii / g_ii)) and
// max |lambda|, three doubles per CTA.
__global__ void __launch_bounds__(256)
    k_refine_norms(int m, const double* __restrict__ G,
                   const double* __restrict__ S, double* __restrict__ part) {
  __shared__ double red[2 * 32];
  __shared__ unsigned long long amax;
  if (threadIdx.x == 0) amax = 0ull;
  __syncthreads();
  double v[2] = {0.0, 0.0};
  unsigned long long mx = 0ull;
  for (size_t e = (size_t)blockIdx.x * 256 + threadIdx.x; e < (size_t)m * m;
       e += (size_t)gridDim.x * 256) {
    const int i = (int)(e % m), j = (int)(e / m);
    double r = -G[e], d = S[e];
    if (i == j) {
      r += 1.0;
      const double lam = S[e] / G[e];
      d -= lam;
      // non-negative doubles order like their bit patterns
      mx = max(mx, (unsigned long long)__double_as_longlong(fabs(lam)));
    }
    v[0] = fma(d, d, v[0]);
    v[1] = fma(r, r, v[1]);
  }
  if (mx) atomicMax(&amax, mx);
  block_sum<2>(v, red);
  if (threadIdx.x == 0) {
    part[3 * blockIdx.x] = v[0];
    part[3 * blockIdx.x + 1] = v[1];
    part[3 * blockIdx.x + 2] = __longlong_as_double((long long)amax);
  }
}

// E of the refinement (see sym_eig), an entry per thread; the nparts partial
// norms are added by every CTA alike. (On one CTA its m^2 FP64 divisions took
// 33 us at m = 64.)
__global__ void __launch_bounds__(256)
    k_refine_eig(int m, const double* __restrict__ G,
                 const double* __restrict__ S, const double* __restrict__ part,
                 int nparts, double* __restrict__ E) {
  __shared__ double sdelta;
  if (threadIdx.x < 32) {
    double a = 0.0, b = 0.0, c = 0.0;
    for (int k = threadIdx.x; k < nparts; k += 32) {
      a += part[3 * k];
      b += part[3 * k + 1];
      c = fmax(c, part[3 * k + 2]);
    }
    a = warp_sum(a);
    b = warp_sum(b);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
      c = fmax(c, __shfl_xor_sync(0xffffffffu, c, o));
    if (threadIdx.x == 0)
      sdelta = 4.0 * rsqrt((double)max(m, 128)) * (sqrt(a) + c * sqrt(b));
  }
  __syncthreads();
  const size_t e = (size_t)blockIdx.x * 256 + threadIdx.x;
  if (e >= (size_t)m * m) return;
  const double delta = sdelta;
  const int i = (int)(e % m), j = (int)(e / m);
  const double lj = S[j + (size_t)j * m] / G[j + (size_t)j * m];
  const double li = S[i + (size_t)i * m] / G[i + (size_t)i * m];
  const double r = (i == j ? 1.0 : 0.0) - G[e];
  const double dl = lj - li;
  const double num = S[e] + lj * r;
  E[e] = (i != j && fabs(dl) > delta && fabs(num) <= 0.01 * fabs(dl))
             ? num / dl
             : 0.5 * r;
}

}  // namespace

void mm_gemm(int m, const double* A, bool trA, const double* B, bool trB,
             double* Cm, double alpha, double beta, cudaStream_t s) {
  GemmOpt o;
  o.cin = Cm;
  mm_launch(m, A, trA, B, trB, Cm, alpha, beta, o, s);
}

void make_A0(int m, const double* Hp, const double* HD, double* A0,
             cudaStream_t s) {
  k_make_A0<<<ceil_div((int64_t)m * m, 256), 256, 0, s>>>(m, Hp, HD, A0);
  TRM_CHECK_LAUNCH();
}


// From this m on the factorisation runs blocked on many CTAs; the
// environment variable TRM_CHOL_BLOCKED_FROM, read once per process,
// overrides the default.
static int chol_blocked_from() {
  static const int v = [] {
    const char* e = std::getenv("TRM_CHOL_BLOCKED_FROM");
    const int d = 256;
    if (!e || !*e) return d;
    const long x = std::strtol(e, nullptr, 10);
    return x > 0 && x <= 4096 ? (int)x : d;
  }();
  return v;
}

// FP64 factor and inverse by correcting FP32 ones: S' (S scaled by powers of
// two to a diagonal near 1), X, two temporaries, Phi, the words of refined_ok,
// k_ref_form's flags (two to a double)
static int ref_ctas(int m) { return ceil_div((int64_t)m * m, 256); }
static size_t refine_elems(int m) {
  return (size_t)5 * m * m + kRefWords + (ref_ctas(m) + 1) / 2;
}

// Does the FP64 factorisation of this size correct an FP32 one (chol_refined)?
// m <= 32 has one panel and gains little (45 us instead of 60): left out.
constexpr int kRefineFrom = 33;
static bool panel_fits(int m);
static bool refines(int m) {
  return m >= kRefineFrom && m < chol_blocked_from() && panel_fits(m);
}

// The largest of what the kernels that may factor this size keep: the padded
// working copy plus the inverse's temporary (one CTA); W, L, X, T and the
// failure flag (blocked: FP64 from chol_blocked_from() on, FP32 above kPanelMax
// too); refine_elems.
size_t chol_work_elems(int m) {
  const size_t mp = (size_t)((m + 31) & ~31);
  size_t n = mp * (mp + 1) + 33 * mp;
  if (m >= chol_blocked_from() || m > kPanelMax)
    n = std::max(n, 4 * mp * mp + 8);
  if (refines(m)) n = std::max(n, refine_elems(m));
  return n;
}

template <typename Tm, bool dev>
static void chol_blocked(int m, const double* S, const double* Bm,
                         const double* Q, const float* Bf, const float* Qf,
                         double* Linv, double* R, IterScalars* sc,
                         double* gwork, cudaStream_t s, const double* lpart,
                         int nlpart) {
  const int mp = (m + 31) & ~31, P = mp / CB;
  const size_t mp2 = (size_t)mp * mp;
  Tm* W = reinterpret_cast<Tm*>(gwork);
  Tm* L = W + mp2;
  Tm* X = L + mp2;
  Tm* T = X + mp2;
  int* bad = reinterpret_cast<int*>(T + mp2);
  if (lpart) {
    k_cb_alpha<<<1, 256, 0, s>>>(m, lpart, nlpart, sc);
    TRM_CHECK_LAUNCH();
  }
  const int fb = (int)std::min<size_t>(ceil_div(mp2, (size_t)256), 1024);
  k_cb_form<Tm, dev><<<fb, 256, 0, s>>>(m, mp, S, Bm, Q, Bf, Qf, sc, W, bad);
  TRM_CHECK_LAUNCH();
  const bool from_S = S != nullptr && !Bm && !Bf;
  for (int p = 0; p < P; ++p) {
    k_cb_diag<Tm, dev><<<1, 256, 0, s>>>(m, mp, p, S, from_S, W, L, X, bad);
    TRM_CHECK_LAUNCH();
    const int t = P - p - 1;
    if (t > 0) {
      k_cb_update<Tm, dev><<<t * (t + 1) / 2, 256, 0, s>>>(mp, p, W, L, X);
      TRM_CHECK_LAUNCH();
    }
  }
  for (int sz = CB; sz < mp; sz *= 2) {
    const dim3 g(ceil_div(mp, 2 * sz), (sz / CB) * (sz / CB));
    k_cb_inv<Tm, dev><<<g, 256, 0, s>>>(mp, sz, 0, L, X, T);
    TRM_CHECK_LAUNCH();
    k_cb_inv<Tm, dev><<<g, 256, 0, s>>>(mp, sz, 1, L, X, T);
    TRM_CHECK_LAUNCH();
  }
  const int ob = (int)std::min<size_t>(ceil_div((size_t)m * m, (size_t)256), 1024);
  k_cb_out<Tm, dev><<<ob, 256, 0, s>>>(m, mp, X, Linv, R, bad, sc);
  TRM_CHECK_LAUNCH();
}

// FP32, m <= kPanelMax: one CTA with everything in shared memory.
template <bool dev>
static void panel_launch(int m, const double* S, const float* Bf,
                         const float* Qf, const PanelOut& out, IterScalars* sc,
                         cudaStream_t s, const double* lpart, int nlpart) {
  static std::atomic<int> done[64] = {};  // per device; any thread may launch
  int dv = 0;
  cudaGetDevice(&dv);
  if (dv < 0 || dv >= 64 || !done[dv].load(std::memory_order_relaxed)) {
    TRM_CUDA(cudaFuncSetAttribute(k_chol_panel<dev>,
                                  cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)panel_smem(kPanelMax)));
    if (dv >= 0 && dv < 64) done[dv].store(1, std::memory_order_relaxed);
  }
  k_chol_panel<dev><<<1, kPanelThreads, panel_smem(m), s>>>(
      m, S, Bf, Qf, out, sc, lpart, nlpart);
  TRM_CHECK_LAUNCH();
}

// FP32 up to this m runs on one CTA out of shared memory (k_chol_panel): at
// m = 256 that is the largest packed copy that fits, and still faster than
// the blocked launches.
static bool panel_fits(int m) {
  return m <= kPanelMax && (m < chol_blocked_from() || m == kPanelMax);
}

// The FP64 factorisation on one CTA is bound by its SM's two FP64 multiply-adds
// a cycle and the pivots' chain. Here the panel kernel's FP32 inverse factor X
// is corrected to FP64 by products, which every SM shares: with F = X S X^T - I
// and Phi the lower triangle of F with half its diagonal,
// (I - Phi) X S X^T (I - Phi)^T = I + O(F^2), so X <- X - Phi X squares the
// error. Two corrections suffice (dev[1], see refined_ok). The rounding errors of
// the products grow with the condition, a little faster than the
// elimination's: max |X - I| < 1/2 (dev[2]) holds it at about 20, within which
// they are smaller (max |X S X^T - I| at m = 64: 3.3e-16 against 5.7e-16 at
// condition 1.5; m = 48, condition 10: 2.8e-16 against 6.0e-16). Otherwise
// nothing is written and k_chol_inv, launched behind it, does its work; it
// returns at once where the result stands. 67 us instead of 166 at m = 64, 101
// instead of 485 at 128. A matrix that is handed on loses what the attempt took:
// 60 and 100 us when it ran to its end, so two tests end it earlier, for
// columns at small angles before it begins (their entry alone is too large) and
// for a large FP32 X before the products; the launches behind them then return
// at once.
static const unsigned long long* chol_refined(int m, const double* S,
                                              const double* Bm, const double* Q,
                                              double* Linv, double* R,
                                              IterScalars* sc, double* gwork,
                                              cudaStream_t s) {
  const size_t mm = (size_t)m * m;
  double* Sp = gwork;
  double* X = Sp + mm;
  double* Xn = X + mm;
  double* T = Xn + mm;
  double* Phi = T + mm;
  auto* dev = reinterpret_cast<unsigned long long*>(Phi + mm);
  auto* hopeless = reinterpret_cast<int*>(dev + kRefWords);
  const int blocks = ref_ctas(m);
  k_ref_form<<<blocks, 256, 0, s>>>(m, S, Bm, Q, sc, Sp, dev, hopeless);
  TRM_CHECK_LAUNCH();
  PanelOut out;
  out.Linv = X;
  out.hopeless = hopeless;
  out.nhopeless = blocks;
  out.stop = dev + kRefStop;
  panel_launch<false>(m, Sp, nullptr, nullptr, out, nullptr, s, nullptr, 0);
  for (int k = 0; k < 2; ++k) {
    GemmOpt a, f, x;
    a.stop = f.stop = x.stop = dev + kRefStop;
    a.tri = kTriA;
    mm_launch(m, X, false, Sp, false, T, 1.0, 0.0, a, s);  // X S'
    f.tri = kTriBt | kTriOut | kPhi;
    f.dev = dev + k;
    mm_launch(m, T, false, X, true, Phi, 1.0, 0.0, f, s);  // X S' X^T
    x.tri = kTriA | kTriB | kTriOut;
    x.cin = X;
    if (k == 1) x.dev = dev + kRefDev2;
    mm_launch(m, Phi, false, X, false, Xn, -1.0, 1.0, x, s);  // X - Phi X
    std::swap(X, Xn);
  }
  k_ref_out<<<blocks, 256, 0, s>>>(m, S, X, dev, Linv, R);
  TRM_CHECK_LAUNCH();
  return dev;
}

template <typename Tm, bool dev>
static void chol_launch(int m, const double* S, const double* Bm,
                        const double* Q, const float* Bf, const float* Qf,
                        double* Linv, double* R, IterScalars* sc,
                        double* gwork, cudaStream_t s,
                        const double* lpart = nullptr, int nlpart = 0) {
  if (m > 1024) throw Error(-1, "chol_inv: m > 1024");
  if constexpr (sizeof(Tm) == 4) {
    if (panel_fits(m)) {
      PanelOut out;
      out.Linv = Linv;
      out.R = R;
      panel_launch<dev>(m, S, Bf, Qf, out, sc, s, lpart, nlpart);
      return;
    }
    chol_blocked<Tm, dev>(m, S, Bm, Q, Bf, Qf, Linv, R, sc, gwork, s, lpart,
                          nlpart);
  } else {
    if (m >= chol_blocked_from()) {
      chol_blocked<Tm, dev>(m, S, Bm, Q, Bf, Qf, Linv, R, sc, gwork, s, lpart,
                            nlpart);
      return;
    }
    const unsigned long long* refined = nullptr;
    if (!dev && refines(m)) {
      if (lpart) {
        k_cb_alpha<<<1, 256, 0, s>>>(m, lpart, nlpart, sc);
        TRM_CHECK_LAUNCH();
        lpart = nullptr;
      }
      refined = chol_refined(m, S, Bm, Q, Linv, R, sc, gwork, s);
    }
    const size_t mp = (size_t)((m + 31) & ~31);
    const size_t bytes = (mp * (mp + 1) + 33 * mp) * sizeof(Tm);
    const bool smem = bytes <= 200 * 1024;
    if (smem) {
      static std::atomic<int> done[64] = {};  // per device; any thread may launch
      int dv = 0;
      cudaGetDevice(&dv);
      if (dv < 0 || dv >= 64 || !done[dv].load(std::memory_order_relaxed)) {
        TRM_CUDA(cudaFuncSetAttribute(k_chol_inv<true>,
                                      cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      200 * 1024));
        if (dv >= 0 && dv < 64) done[dv].store(1, std::memory_order_relaxed);
      }
    }
    if (smem)
      k_chol_inv<true><<<1, kCholThreads, bytes, s>>>(
          m, S, Bm, Q, Linv, R, sc, nullptr, lpart, nlpart, refined);
    else
      k_chol_inv<false><<<1, kCholThreads, 0, s>>>(
          m, S, Bm, Q, Linv, R, sc, gwork, lpart, nlpart, refined);
    TRM_CHECK_LAUNCH();
  }
}

template <typename Tm>
void chol_inv(int m, const double* S, double* Linv, double* R, IterScalars* sc,
              double* gwork, cudaStream_t s) {
  chol_launch<Tm, false>(m, S, nullptr, nullptr, nullptr, nullptr, Linv, R,
                         sc, gwork, s);
}

// k-splits of the line terms: about 64 CTAs when the m x m tiles are few
// (partials: 4 doubles per CTA, at most 4 ceil(m/32)^2 * 4 in all)
static int line_ksplit(int m) {
  const int t = ceil_div(m, 32);
  const int ks = std::min(std::min(t, 4), std::max(1, 64 / (t * t)));
  return std::max(1, ks);
}

void line_factor(int m, const double* Hp, const double* HD, const double* Bm,
                 const double* Q, const double* hpd, int hpd_stride,
                 const double* tr_parts, int n_tr_parts, const double* W,
                 double* R, IterScalars* sc, double* gwork, double* part,
                 cudaStream_t s) {
  const int t = ceil_div(m, 32);
  const int ksplit = line_ksplit(m);
  k_line_terms<double><<<dim3(t, t, ksplit), 1024, 0, s>>>(
      m, Hp, HD, Bm, Q, hpd, hpd_stride, tr_parts, n_tr_parts, W, part);
  TRM_CHECK_LAUNCH();
  // the factorisation kernel takes the line step from the partials first
  chol_launch<double, false>(m, nullptr, Bm, Q, nullptr, nullptr, nullptr, R, sc,
                             gwork, s, part, t * t * ksplit);
}

// The FP32 path with the m x m inputs already in FP32 (copies the Gram sums
// write): no FP64 conversion in the line terms or the factorisation.
bool line_factor32(int m, const float* Hp, const double* HD, const float* Bm,
                   const float* Q, const double* hpd, int hpd_stride,
                   const double* tr_parts, int n_tr_parts, const float* W,
                   double* R, IterScalars* sc, double* gwork, double* part,
                   cudaStream_t s, float* split, int split_ldm,
                   bool split_diag) {
  const int t = ceil_div(m, 32);
  const int ksplit = line_ksplit(m);
  k_line_terms<float><<<dim3(t, t, ksplit), 1024, 0, s>>>(
      m, Hp, HD, Bm, Q, hpd, hpd_stride, tr_parts, n_tr_parts, W, part);
  TRM_CHECK_LAUNCH();
  if (split && panel_fits(m)) {
    PanelOut out;
    out.split = split;
    out.ldm = split_ldm;
    out.split_diag = split_diag ? 1 : 0;
    panel_launch<true>(m, nullptr, Bm, Q, out, sc, s, part, t * t * ksplit);
    return true;
  }
  chol_launch<float, true>(m, nullptr, nullptr, nullptr, Bm, Q, nullptr, R, sc,
                           gwork, s, part, t * t * ksplit);
  return false;
}

template <typename T>
static void jacobi_launch(int m, const double* A, const double* Z0, double* w,
                          double* Z, T* Aw, T* Zw, int* info, int max_sweeps,
                          T rot_tol, T abs_c, T conv_tol, cudaStream_t s) {
  const size_t bytes = (size_t)m * (m + 1) * sizeof(T);
  const bool smem = bytes <= 200 * 1024;
  if (smem) {
    static std::atomic<int> done[64] = {};  // per device; any thread may launch
    int dv = 0;
    cudaGetDevice(&dv);
    if (dv < 0 || dv >= 64 || !done[dv].load(std::memory_order_relaxed)) {
      TRM_CUDA(cudaFuncSetAttribute(k_jacobi<T>,
                                    cudaFuncAttributeMaxDynamicSharedMemorySize,
                                    200 * 1024));
      if (dv >= 0 && dv < 64) done[dv].store(1, std::memory_order_relaxed);
    }
  }
  k_jacobi<T><<<1, 1024, smem ? bytes : 0, s>>>(m, A, Aw, Zw, Z0, w, Z, info,
                                                max_sweeps, rot_tol, abs_c,
                                                conv_tol, smem ? 1 : 0);
  TRM_CHECK_LAUNCH();
}

// 8 m x m matrices, 2 x 4 deviations, the partial norms
constexpr int kNormParts = 64;
size_t sym_eig_work_doubles(int m) {
  return (size_t)8 * m * m + 8 + 3 * kNormParts;
}

void newton_schulz(int m, double*& X, double*& Xn, double* G,
                   unsigned long long* dev, int steps, cudaStream_t s) {
  for (int k = 0; k < steps; ++k) {
    GemmOpt g;
    g.skip = k ? dev + k - 1 : nullptr;
    g.dev = dev + k;  // stays 0 when skipped: so are all later ones
    mm_launch(m, X, true, X, false, G, 1.0, 0.0, g, s);
    GemmOpt h;
    h.cin = X;
    h.skip = g.skip;
    mm_launch(m, X, false, G, false, Xn, -0.5, 1.5, h, s);
    std::swap(X, Xn);
  }
}

// FP32 Jacobi sweeps (the FP64 pipe is 1/64 of the FP32 one); then twice:
// one FP64 refinement of the eigenvectors by matrix products on many CTAs,
// and four Newton-Schulz steps X <- X (3 I - X^T X) / 2 (the refinement is
// first order: where it splits close pairs it leaves X non-orthonormal by
// the square of its step, and X^T A X would then not be similar to A; the
// quadratically convergent steps bring that to FP64 rounding from up to
// ~0.1); then FP64 Jacobi on X^T A X, nearly diagonal, which rotates
// only the pairs still coupled above FP64 product noise (clusters) and
// accumulates onto X.
void sym_eig(int m, const double* A, double* w, double* Z, double* work,
             int* info, cudaStream_t s) {
  if (m > 1024) throw Error(-1, "sym_eig: m > 1024");
  const size_t mm = (size_t)m * m;
  double* X = work;
  double* T = work + mm;
  double* Sx = work + 2 * mm;
  double* G = work + 3 * mm;
  double* E = work + 4 * mm;
  double* Xn = work + 5 * mm;
  double* jw = work + 6 * mm;  // Jacobi work copies (2 m^2 of its type)
  // FP32 sweeps until no coupling above 4e-7 of its pair's diagonal plus
  // 1e-6 ||A||_F is left
  jacobi_launch<float>(m, A, nullptr, w, X, reinterpret_cast<float*>(jw),
                       reinterpret_cast<float*>(jw) + mm, info, 20, 4e-7f,
                       1e-6f, 0.0f, s);
  constexpr int kNs = 4;
  auto* dev = reinterpret_cast<unsigned long long*>(work + 8 * mm);
  double* norms = work + 8 * mm + 2 * kNs;
  const int nparts = std::min(ceil_div((int64_t)mm, 1024), kNormParts);
  TRM_CUDA(cudaMemsetAsync(dev, 0, 2 * kNs * sizeof(*dev), s));
  for (int it = 0; it < 2; ++it) {
    mm_gemm(m, A, false, X, false, T, 1.0, 0.0, s);   // A X
    mm_gemm(m, X, true, T, false, Sx, 1.0, 0.0, s);   // X^T A X
    mm_gemm(m, X, true, X, false, G, 1.0, 0.0, s);    // X^T X
    k_refine_norms<<<nparts, 256, 0, s>>>(m, G, Sx, norms);
    TRM_CHECK_LAUNCH();
    k_refine_eig<<<ceil_div((int64_t)mm, 256), 256, 0, s>>>(m, G, Sx, norms,
                                                            nparts, E);
    TRM_CHECK_LAUNCH();
    GemmOpt o;
    o.cin = X;
    mm_launch(m, X, false, E, false, Xn, 1.0, 1.0, o, s);  // X + X E
    std::swap(X, Xn);
    newton_schulz(m, X, Xn, G, dev + it * kNs, kNs, s);
  }
  mm_gemm(m, A, false, X, false, T, 1.0, 0.0, s);
  mm_gemm(m, X, true, T, false, Sx, 1.0, 0.0, s);
  jacobi_launch<double>(m, Sx, X, w, Z, jw, jw + mm, info, 8, 1e-13, 1e-15,
                        0.0, s);
}

template void chol_inv<float>(int, const double*, double*, double*,
                              IterScalars*, double*, cudaStream_t);
template void chol_inv<double>(int, const double*, double*, double*,
                               IterScalars*, double*, cudaStream_t);

}  // namespace trm
