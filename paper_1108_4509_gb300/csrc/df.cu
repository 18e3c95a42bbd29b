// Double-float ("FP32 pair") arithmetic for the FP64-accuracy steps of the
// MP2 phase (Sec. 2.2: H C, the energy terms H_D and X' = X - C diag(H_D)).
//
// GB300 runs FP64 at 1/64 of its FP32 rate, and the FP64 stencil was bound
// by that pipe. Here a value is held as hi + lo with hi = fl32(v) and
// lo = fl32(v - hi) (|lo| <= ulp(hi)/2, about 48 significant bits), and
// sums and products use the error-free transformations of Knuth (TwoSum)
// and Dekker/Kahan (TwoProduct with a fused multiply-add), so the results
// carry a relative error of a few units of 2^-48 of the magnitudes involved
// — far below what E_G at 1e-10 and residuals at 1e-10 need — while every
// operation runs on the FP32 pipe. No FP64 instruction is executed per
// element, except once per thread when an FP64 scalar is split.
#include <type_traits>

#include "dfmath.cuh"
#include "ops.cuh"

namespace trm {

namespace {

// hi + lo in FP64, widened on the integer pipe: one FP64 instruction (the
// sum) instead of three.
__device__ __forceinline__ double widen(float f) {
  const uint32_t u = __float_as_uint(f);
  if ((u & 0x7F800000u) == 0 && (u & 0x7FFFFFu)) return (double)f;
  return to_f64(f);
}

// Bound by memory at 16 bytes an element. With the conversion instructions
// they were bound by the FP64 pipe (48^3 x 128: split 103, join 78 us).
__global__ void __launch_bounds__(256)
    k_split_df(int64_t n, const double* __restrict__ x, float* __restrict__ hi,
               float* __restrict__ lo, int vec) {
  const int64_t t0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t step = (int64_t)gridDim.x * blockDim.x;
  if (vec) {
    for (int64_t i = t0; i < (n >> 2); i += step) {
      const double2 a = reinterpret_cast<const double2*>(x)[2 * i];
      const double2 b = reinterpret_cast<const double2*>(x)[2 * i + 1];
      const F2 v0 = df_of_bits(a.x), v1 = df_of_bits(a.y),
               v2 = df_of_bits(b.x), v3 = df_of_bits(b.y);
      reinterpret_cast<float4*>(hi)[i] = make_float4(v0.h, v1.h, v2.h, v3.h);
      reinterpret_cast<float4*>(lo)[i] = make_float4(v0.l, v1.l, v2.l, v3.l);
    }
  } else {
    for (int64_t i = t0; i < n; i += step) {
      const F2 v = df_of_bits(x[i]);
      hi[i] = v.h;
      lo[i] = v.l;
    }
  }
}

__global__ void __launch_bounds__(256)
    k_join_df(int64_t n, const float* __restrict__ hi,
              const float* __restrict__ lo, double* __restrict__ x, int vec) {
  const int64_t t0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t step = (int64_t)gridDim.x * blockDim.x;
  if (vec) {
    // two entries a thread: 16-byte stores next to each other (four entries
    // as two stores 32 bytes apart wrote half sectors, at half the rate)
#pragma unroll 4
    for (int64_t i = t0; i < (n >> 1); i += step) {
      const float2 h = reinterpret_cast<const float2*>(hi)[i];
      const float2 l = reinterpret_cast<const float2*>(lo)[i];
      reinterpret_cast<double2*>(x)[i] =
          make_double2(widen(h.x) + widen(l.x), widen(h.y) + widen(l.y));
    }
  } else {
    for (int64_t i = t0; i < n; i += step) x[i] = widen(hi[i]) + widen(lo[i]);
  }
}

constexpr int kCols = 4;  // columns per CTA (grid.y walks column groups)

// ---------------------------------------------------------------------------
// X = H C for the stencil operator as a register z-march (see k_stencil_zm): a
// thread owns VW (2 or 1) consecutive x points of one column and walks a chunk
// of planes with the 2R + 1 pairs of each along z in registers. The FP32 pipe is
// what bounds it, so the pairs are summed without intermediate normalisations:
// the hi parts by TwoSum, the lo parts and rounding errors plainly, the three
// products as (fl, error) by fused multiply-adds, one renormalisation at the
// end: about 112 operations a point, the errors a few units of 2^-48 of the
// magnitudes as before. The column dots H_D = c_j . (H c)_j of
// Fig. EGFIG step (2) are formed from the pairs in registers (double-float per
// thread and warp, one FP64 add per warp): CTA (t, u) writes
// dots[(u gridDim.x + t) ncols + column].
// It replaces kernels that took the z neighbours through L2 with two CTAs per
// SM (98 registers): 160 us at 48^3 x 128 and 4.94 ms at 96^3 x 512, now 113 us
// and 2.94 ms. The pairs' arithmetic is the bound (0.30 of the copy bandwidth).
// ---------------------------------------------------------------------------
// s + l += (h, l) of a neighbour
__device__ __forceinline__ void acc_add(F2& a, float h, float l) {
  const F2 t = two_sum(a.h, h);
  a.h = t.h;
  a.l += t.l + l;
}
// p + e = a b with |e| at 2^-48 of the product (not renormalised)
__device__ __forceinline__ F2 prod_df(F2 a, F2 b) {
  const float p = a.h * b.h;
  float e = fmaf(a.h, b.h, -p);
  e = fmaf(a.h, b.l, e);
  return {p, fmaf(a.l, b.h, e)};
}
template <int VW>
struct PairV {
  float h[VW], l[VW];
};
template <int VW>
__device__ __forceinline__ PairV<VW> ldp(const float* h, const float* l,
                                         int64_t o, bool in) {
  PairV<VW> v;
  if constexpr (VW == 2) {
    const float2 z = make_float2(0.f, 0.f);
    const float2 a = in ? __ldg(reinterpret_cast<const float2*>(h + o)) : z;
    const float2 b = in ? __ldg(reinterpret_cast<const float2*>(l + o)) : z;
    v.h[0] = a.x; v.h[1] = a.y;
    v.l[0] = b.x; v.l[1] = b.y;
  } else {
    v.h[0] = in ? __ldg(h + o) : 0.f;
    v.l[0] = in ? __ldg(l + o) : 0.f;
  }
  return v;
}

template <int R, int VW>
__global__ void __launch_bounds__(256, 3)
    k_stencil_df(StencilOp st, int64_t ld, const float* __restrict__ dh,
                 const float* __restrict__ dl, const float* __restrict__ Ch,
                 const float* __restrict__ Cl, float* __restrict__ Xh,
                 float* __restrict__ Xl, int ncols, int zc, int pack,
                 double* __restrict__ dots) {
  __shared__ double red[8];
  const int nx = st.nx, ny = st.ny, nz = st.nz, nxq = nx / VW;
  int p, z0;  // group in the plane, first plane
  const bool active = zm_place(nxq * ny, nz, zc, pack, p, z0);
  const int x0 = active ? VW * (p % nxq) : 0, y = active ? p / nxq : 0;
  const int col = blockIdx.z;
  const int z1 = min(nz, z0 + zc);
  const int64_t sz = (int64_t)nx * ny;
  const int64_t rowoff = (int64_t)y * nx + x0;
  const float* ch = Ch + (int64_t)col * ld + rowoff;
  const float* cl = Cl + (int64_t)col * ld + rowoff;
  const bool ym1 = y >= 1, yp1 = y + 1 < ny, ym2 = y >= 2, yp2 = y + 2 < ny;
  const F2 c1 = {st.c1h, st.c1l}, c2 = {st.c2h, st.c2l};
  PairV<VW> q[2 * R + 2];  // planes z - R .. z + R, and z + R + 1 in flight
#pragma unroll
  for (int k = 0; k < 2 * R + 1; ++k) {
    const int pz = z0 - R + k;
    q[k] = ldp<VW>(ch, cl, pz * sz, active && pz >= 0 && pz < nz);
  }
  F2 dacc = {0.f, 0.f};
  for (int z = z0; z < z1; ++z) {
    const int64_t o = z * sz;
    q[2 * R + 1] = ldp<VW>(ch, cl, o + (R + 1) * sz,
                           active && z + R + 1 < nz && z + 1 < z1);
    if (active) {
      // the row's values x0 - 2 .. x0 + VW + 1
      float eh[VW + 4], el[VW + 4];
#pragma unroll
      for (int k = 0; k < VW; ++k) {
        eh[k + 2] = q[R].h[k];
        el[k + 2] = q[R].l[k];
      }
      if constexpr (VW == 2) {
        const PairV<2> a = ldp<2>(ch, cl, o - 2, x0 >= 2);
        const PairV<2> b = ldp<2>(ch, cl, o + 2, x0 + 2 < nx);
        eh[0] = a.h[0]; eh[1] = a.h[1]; eh[4] = b.h[0]; eh[5] = b.h[1];
        el[0] = a.l[0]; el[1] = a.l[1]; el[4] = b.l[0]; el[5] = b.l[1];
      } else {
        const PairV<1> a = ldp<1>(ch, cl, o - 1, x0 >= 1);
        const PairV<1> b = ldp<1>(ch, cl, o + 1, x0 + 1 < nx);
        eh[1] = a.h[0]; eh[3] = b.h[0];
        el[1] = a.l[0]; el[3] = b.l[0];
        if (R == 2) {
          const PairV<1> a2 = ldp<1>(ch, cl, o - 2, x0 >= 2);
          const PairV<1> b2 = ldp<1>(ch, cl, o + 2, x0 + 2 < nx);
          eh[0] = a2.h[0]; eh[4] = b2.h[0];
          el[0] = a2.l[0]; el[4] = b2.l[0];
        }
      }
      const PairV<VW> d = ldp<VW>(dh, dl, o + rowoff, true);
      F2 s1[VW], s2[VW];
      {
        const PairV<VW> a = ldp<VW>(ch, cl, o - nx, ym1);
        const PairV<VW> b = ldp<VW>(ch, cl, o + nx, yp1);
#pragma unroll
        for (int k = 0; k < VW; ++k) {
          s1[k] = F2{a.h[k], a.l[k]};
          acc_add(s1[k], b.h[k], b.l[k]);
          acc_add(s1[k], q[R - 1].h[k], q[R - 1].l[k]);
          acc_add(s1[k], q[R + 1].h[k], q[R + 1].l[k]);
          acc_add(s1[k], eh[k + 1], el[k + 1]);
          acc_add(s1[k], eh[k + 3], el[k + 3]);
        }
      }
      if (R == 2) {
        const PairV<VW> a = ldp<VW>(ch, cl, o - 2 * nx, ym2);
        const PairV<VW> b = ldp<VW>(ch, cl, o + 2 * nx, yp2);
#pragma unroll
        for (int k = 0; k < VW; ++k) {
          s2[k] = F2{a.h[k], a.l[k]};
          acc_add(s2[k], b.h[k], b.l[k]);
          acc_add(s2[k], q[0].h[k], q[0].l[k]);
          acc_add(s2[k], q[2 * R].h[k], q[2 * R].l[k]);
          acc_add(s2[k], eh[k], el[k]);
          acc_add(s2[k], eh[k + 4], el[k + 4]);
        }
      }
      float oh[VW], ol[VW];
#pragma unroll
      for (int k = 0; k < VW; ++k) {
        const F2 c = {q[R].h[k], q[R].l[k]};
        const F2 a = prod_df(F2{d.h[k], d.l[k]}, c);
        const F2 b = prod_df(c1, s1[k]);
        F2 t = two_sum(a.h, b.h);
        t.l += a.l + b.l;
        if (R == 2) {
          const F2 e = prod_df(c2, s2[k]);
          const F2 u = two_sum(t.h, e.h);
          t.h = u.h;
          t.l += u.l + e.l;
        }
        t = quick_two_sum(t.h, t.l);
        oh[k] = t.h;
        ol[k] = t.l;
        const F2 w = prod_df(c, t);
        const F2 u = two_sum(dacc.h, w.h);
        dacc.h = u.h;
        dacc.l += u.l + w.l;
      }
      const int64_t x = (int64_t)col * ld + rowoff + o;
      if constexpr (VW == 2) {
        *reinterpret_cast<float2*>(Xh + x) = make_float2(oh[0], oh[1]);
        *reinterpret_cast<float2*>(Xl + x) = make_float2(ol[0], ol[1]);
      } else {
        Xh[x] = oh[0];
        Xl[x] = ol[0];
      }
      dacc = quick_two_sum(dacc.h, dacc.l);
    }
#pragma unroll
    for (int k = 0; k < 2 * R + 1; ++k) q[k] = q[k + 1];
  }
  {
    F2 w = dacc;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
      w = df_add(w, F2{__shfl_xor_sync(0xffffffffu, w.h, o),
                       __shfl_xor_sync(0xffffffffu, w.l, o)});
    if ((threadIdx.x & 31) == 0)
      red[threadIdx.x >> 5] = to_f64(w.h) + to_f64(w.l);
    __syncthreads();
    if (threadIdx.x == 0) {
      double t = 0.0;
      for (int k = 0; k < (int)(blockDim.x + 31) / 32; ++k) t += red[k];
      dots[((size_t)blockIdx.y * gridDim.x + blockIdx.x) * ncols + col] = t;
    }
  }
}

// X = H C for a CSR operator (values split into hi + lo at creation), one row
// per thread and kCols columns together: an entry's index and value are read
// once for them, the products are added as in k_stencil_df (hi parts by TwoSum,
// the rest plainly), and the column dots c_j . (H c)_j: CTA b writes
// dots[b ncols + column]. One column at a time with normalised sums it took 44
// instructions an entry (420 us at N = 48^3, 13 entries a row, 128 columns) and
// the dots 43 us in a kernel of their own; now 252 us with the dots.
__global__ void __launch_bounds__(256)
    k_csr_df(int64_t N, int64_t ld, const int32_t* __restrict__ rowptr,
             const int32_t* __restrict__ cols, const float* __restrict__ vh,
             const float* __restrict__ vl, const float* __restrict__ Ch,
             const float* __restrict__ Cl, float* __restrict__ Xh,
             float* __restrict__ Xl, int ncols, double* __restrict__ dots) {
  __shared__ double red[kCols][8];
  const int64_t r0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const bool valid = r0 < N;
  const int64_t r = valid ? r0 : 0;
  const int b = valid ? rowptr[r] : 0, e = valid ? rowptr[r + 1] : 0;
  const int cb = blockIdx.y * kCols, nc = min(kCols, ncols - cb);
  const float* ph[kCols];
  const float* pl[kCols];
  F2 acc[kCols];
#pragma unroll
  for (int q = 0; q < kCols; ++q) {
    const int64_t o = (int64_t)(cb + min(q, nc - 1)) * ld;
    ph[q] = Ch + o;
    pl[q] = Cl + o;
    acc[q] = F2{0.f, 0.f};
  }
  auto row = [&](auto full) {
#pragma unroll 2
    for (int k = b; k < e; ++k) {
      const int j = cols[k];
      const F2 v = {vh[k], vl[k]};
#pragma unroll
      for (int q = 0; q < kCols; ++q)
        if (decltype(full)::value || q < nc) {
          const F2 t = prod_df(v, F2{__ldg(ph[q] + j), __ldg(pl[q] + j)});
          acc_add(acc[q], t.h, t.l);
          acc[q] = quick_two_sum(acc[q].h, acc[q].l);
        }
    }
  };
  if (nc == kCols)
    row(std::true_type{});
  else
    row(std::false_type{});
  F2 d[kCols];
#pragma unroll
  for (int q = 0; q < kCols; ++q) {
    d[q] = F2{0.f, 0.f};
    if (valid && q < nc) {
      const F2 t = quick_two_sum(acc[q].h, acc[q].l);
      const int64_t o = (int64_t)(cb + q) * ld + r;
      Xh[o] = t.h;
      Xl[o] = t.l;
      d[q] = df_mul(F2{ph[q][r], pl[q][r]}, t);
    }
  }
  {
#pragma unroll
    for (int q = 0; q < kCols; ++q) {
      F2 w = d[q];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1)
        w = df_add(w, F2{__shfl_xor_sync(0xffffffffu, w.h, o),
                         __shfl_xor_sync(0xffffffffu, w.l, o)});
      if ((threadIdx.x & 31) == 0)
        red[q][threadIdx.x >> 5] = to_f64(w.h) + to_f64(w.l);
    }
    __syncthreads();
    if ((int)threadIdx.x < nc) {
      double t = red[threadIdx.x][0];
#pragma unroll
      for (int w = 1; w < 8; ++w) t += red[threadIdx.x][w];
      dots[(size_t)blockIdx.x * ncols + cb + threadIdx.x] = t;
    }
  }
}

// X32 = fl32(X - C diag(H_D))
__global__ void k_xprime_df(int64_t N, const float* __restrict__ Ch,
                            const float* __restrict__ Cl,
                            const float* __restrict__ Xh,
                            const float* __restrict__ Xl,
                            const double* __restrict__ HD,
                            float* __restrict__ X32) {
  const int j = blockIdx.y;
  const F2 h = df_of(-HD[j]);
  const int64_t off = (int64_t)j * N;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < N;
       i += (int64_t)gridDim.x * blockDim.x) {
    const F2 t = df_mul(F2{Ch[off + i], Cl[off + i]}, h);
    X32[off + i] = df_add(F2{Xh[off + i], Xl[off + i]}, t).h;
  }
}

// The same on 16-byte vectors (N % 4 == 0, aligned blocks).
__global__ void k_xprime_df4(int64_t N, const float4* __restrict__ Ch,
                             const float4* __restrict__ Cl,
                             const float4* __restrict__ Xh,
                             const float4* __restrict__ Xl,
                             const double* __restrict__ HD,
                             float4* __restrict__ X32) {
  const int j = blockIdx.y;
  const F2 h = df_of(-HD[j]);
  const int64_t n4 = N >> 2, off = (int64_t)j * n4;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n4;
       i += (int64_t)gridDim.x * blockDim.x) {
    const float4 a = Ch[off + i], b = Cl[off + i], c = Xh[off + i],
                 d = Xl[off + i];
    float4 o;
    o.x = df_add(F2{c.x, d.x}, df_mul(F2{a.x, b.x}, h)).h;
    o.y = df_add(F2{c.y, d.y}, df_mul(F2{a.y, b.y}, h)).h;
    o.z = df_add(F2{c.z, d.z}, df_mul(F2{a.z, b.z}, h)).h;
    o.w = df_add(F2{c.w, d.w}, df_mul(F2{a.w, b.w}, h)).h;
    X32[off + i] = o;
  }
}

int grid_1d(int64_t n) {
  const int64_t g = (n + 255) / 256;
  return (int)(g < 1 ? 1 : (g > 8 * 4096 ? 8 * 4096 : g));
}

}  // namespace

// whole quads at 16-byte aligned addresses?
static int quads(int64_t n, const void* a, const void* b, const void* c) {
  return n % 4 == 0 && ((reinterpret_cast<uintptr_t>(a) |
                         reinterpret_cast<uintptr_t>(b) |
                         reinterpret_cast<uintptr_t>(c)) & 15) == 0;
}

void split_df(const double* x, float* hi, float* lo, int64_t n,
              cudaStream_t s) {
  const int vec = quads(n, x, hi, lo);
  k_split_df<<<grid_1d(vec ? n / 4 : n), 256, 0, s>>>(n, x, hi, lo, vec);
  TRM_CHECK_LAUNCH();
}

void join_df(const float* hi, const float* lo, double* x, int64_t n,
             cudaStream_t s) {
  const int vec = quads(n, x, hi, lo);
  k_join_df<<<grid_1d(vec ? n / 4 : n), 256, 0, s>>>(n, hi, lo, x, vec);
  TRM_CHECK_LAUNCH();
}

namespace {

template <int R, int VW>
int launch_df(const Operator& op, const float* Ch, const float* Cl, float* Xh,
              float* Xl, int ncols, double* dots, cudaStream_t s) {
  const StencilOp st = zm_axes(op.st);
  const ZmShape z =
      zm_shape(st, op.N, ncols, VW, (int)apply_h_dots_doubles(op, 1));
  k_stencil_df<R, VW><<<dim3(z.tiles, z.chunks, ncols), z.threads, 0, s>>>(
      st, op.ld, op.diag32, op.diaglo, Ch, Cl, Xh, Xl, ncols, z.zc,
      z.pack, dots);
  TRM_CHECK_LAUNCH();
  return z.tiles * z.chunks;  // partial dots per column
}

int stencil_df(const Operator& op, const float* Ch, const float* Cl, float* Xh,
               float* Xl, int ncols, double* dots, cudaStream_t s) {
  if (ncols > 65535) throw Error(-1, "too many columns for one launch");
  const uintptr_t a = reinterpret_cast<uintptr_t>(Ch) |
                      reinterpret_cast<uintptr_t>(Cl) |
                      reinterpret_cast<uintptr_t>(Xh) |
                      reinterpret_cast<uintptr_t>(Xl) |
                      reinterpret_cast<uintptr_t>(op.diag32) |
                      reinterpret_cast<uintptr_t>(op.diaglo);
  // (short rows of a one-plane grid: one point a thread fills the warps better)
  const bool two = (op.st.nx | op.ld) % 2 == 0 && a % 8 == 0 &&
                   !(op.st.nz == 1 && op.st.nx < 64);
  if (op.st.radius == 1)
    return two ? launch_df<1, 2>(op, Ch, Cl, Xh, Xl, ncols, dots, s)
               : launch_df<1, 1>(op, Ch, Cl, Xh, Xl, ncols, dots, s);
  return two ? launch_df<2, 2>(op, Ch, Cl, Xh, Xl, ncols, dots, s)
             : launch_df<2, 1>(op, Ch, Cl, Xh, Xl, ncols, dots, s);
}

int csr_df(const Operator& op, const float* Ch, const float* Cl, float* Xh,
           float* Xl, int ncols, double* dots, cudaStream_t s) {
  const int gy = ceil_div(ncols, kCols);
  if (gy > 65535) throw Error(-1, "too many columns for one launch");
  const dim3 grid(ceil_div(op.N, 256), gy);
  k_csr_df<<<grid, 256, 0, s>>>(op.N, op.ld, op.csr.rowptr, op.csr.cols,
                                      op.csr.valshi, op.csr.valslo, Ch, Cl, Xh,
                                      Xl, ncols, dots);
  TRM_CHECK_LAUNCH();
  return (int)grid.x;
}

}  // namespace

int apply_h_df_dots(const Operator& op, const float* Ch, const float* Cl,
                    float* Xh, float* Xl, int ncols, double* dots,
                    cudaStream_t s) {
  if (ncols <= 0) return 0;
  return op.kind == 0 ? stencil_df(op, Ch, Cl, Xh, Xl, ncols, dots, s)
                      : csr_df(op, Ch, Cl, Xh, Xl, ncols, dots, s);
}

void xprime_df(int64_t N, int m, const float* Ch, const float* Cl,
               const float* Xh, const float* Xl, const double* HD, float* X32,
               cudaStream_t s) {
  int gx = ceil_div(N, 256 * 4);
  gx = gx < 1 ? 1 : (gx > 4096 ? 4096 : gx);
  if (N % 4 == 0 &&
      ((reinterpret_cast<uintptr_t>(Ch) | reinterpret_cast<uintptr_t>(Cl) |
        reinterpret_cast<uintptr_t>(Xh) | reinterpret_cast<uintptr_t>(Xl) |
        reinterpret_cast<uintptr_t>(X32)) & 15) == 0) {
    k_xprime_df4<<<dim3(gx, m), 256, 0, s>>>(
        N, reinterpret_cast<const float4*>(Ch), reinterpret_cast<const float4*>(Cl),
        reinterpret_cast<const float4*>(Xh), reinterpret_cast<const float4*>(Xl),
        HD, reinterpret_cast<float4*>(X32));
    TRM_CHECK_LAUNCH();
    return;
  }
  k_xprime_df<<<dim3(gx, m), 256, 0, s>>>(N, Ch, Cl, Xh, Xl, HD, X32);
  TRM_CHECK_LAUNCH();
}

}  // namespace trm
