// H applied to a block of columns: X = H C (Fig. EGFIG, step (1)).
//
// Stencil operators: H = t (T_x (+) T_y (+) T_z) + diag(V) on a Dirichlet grid,
// x fastest. Every column is one grid function; a thread owns four consecutive
// x points of one (y, z) row and walks a few columns, so the grid-index work
// and the diagonal are shared across columns and every access is a 16-byte
// vector load (x neighbours come from the vectors left and right of it).
// CSR operators: one thread per row takes the columns of its column group
// together.
#include <algorithm>
#include <atomic>
#include <cstdlib>
#include <type_traits>
#include <cstring>
#include <map>
#include <mutex>
#include <tuple>

#include "dfmath.cuh"
#include "ops.cuh"
#include "tc.cuh"

namespace trm {

namespace {

template <typename T>
struct V4 {
  T v[4];
};

__device__ __forceinline__ V4<float> ld4(const float* p) {
  float4 a = __ldg(reinterpret_cast<const float4*>(p));
  return {{a.x, a.y, a.z, a.w}};
}
__device__ __forceinline__ V4<double> ld4(const double* p) {
  double2 a = __ldg(reinterpret_cast<const double2*>(p));
  double2 b = __ldg(reinterpret_cast<const double2*>(p) + 1);
  return {{a.x, a.y, b.x, b.y}};
}
__device__ __forceinline__ void st4(float* p, const V4<float>& v) {
  *reinterpret_cast<float4*>(p) = make_float4(v.v[0], v.v[1], v.v[2], v.v[3]);
}
__device__ __forceinline__ void st4(double* p, const V4<double>& v) {
  reinterpret_cast<double2*>(p)[0] = make_double2(v.v[0], v.v[1]);
  reinterpret_cast<double2*>(p)[1] = make_double2(v.v[2], v.v[3]);
}

template <typename T>
__device__ __forceinline__ const T* diag_ptr(const double* d64,
                                             const float* d32);
template <>
__device__ __forceinline__ const float* diag_ptr<float>(const double*,
                                                        const float* d32) {
  return d32;
}
template <>
__device__ __forceinline__ const double* diag_ptr<double>(const double* d64,
                                                          const float*) {
  return d64;
}

// Columns per CTA (grid.y walks column groups).
constexpr int kCpb = 4;

// Column dot products sum_i X_ic Y_ic fused into H X (Fig. EGFIG steps
// (2), (3) read exactly the block pair this kernel holds): every warp adds
// its lanes' products per column into red[q][warp]; after the column loop
// the CTA's 8 warp sums are added in a fixed order and written to
// dots[blockIdx.x * ncols + c].
template <typename T>
__device__ __forceinline__ void warp_dot(T d, double (*red)[8], int q) {
  d = warp_sum(d);
  if ((threadIdx.x & 31) == 0) red[q][threadIdx.x >> 5] = to_f64(d);
}
__device__ __forceinline__ void write_dots(double (*red)[8], double* dots,
                                           int cb, int ncols) {
  __syncthreads();
  if (threadIdx.x < kCpb && cb + (int)threadIdx.x < ncols) {
    double t = red[threadIdx.x][0];
#pragma unroll
    for (int w = 1; w < 8; ++w) t += red[threadIdx.x][w];
    dots[(size_t)blockIdx.x * ncols + cb + threadIdx.x] = t;
  }
}

// Four x points per thread; requires nx % 4 == 0. The kernel waits on its
// neighbour loads (L1/L2 latency, not bandwidth), so the FP32 instances are
// held to 48 registers for five 256-thread CTAs per SM (measured: 12 % faster
// at 48^3 and 21 % at 96^3, m = 128, than at 63 registers and four CTAs).
template <typename T, int R, bool DOTS>
__global__ void __launch_bounds__(256, sizeof(T) == 4 ? 5 : 1)
    k_stencil_v4(StencilOp st, int64_t N, const double* __restrict__ d64,
                 const float* __restrict__ d32, const T* __restrict__ X,
                 T* __restrict__ Y, int ncols, double* __restrict__ dots) {
  const int64_t nv = N >> 2;
  const int64_t v0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const bool valid = v0 < nv;
  if (!DOTS && !valid) return;  // with DOTS every thread joins the sums
  const int64_t v = valid ? v0 : 0;
  __shared__ double red[kCpb][8];
  const int nxv = st.nx >> 2;
  const int xv = (int)(v % nxv);
  const int64_t yz = v / nxv;
  const int y = (int)(yz % st.ny);
  const int z = (int)(yz / st.ny);
  const int64_t i0 = v << 2;
  const int64_t sy = st.nx, sz = (int64_t)st.nx * st.ny;
  const bool xl = xv > 0, xr = xv + 1 < nxv;
  const bool ym1 = y >= 1, yp1 = y + 1 < st.ny;
  const bool zm1 = z >= 1, zp1 = z + 1 < st.nz;
  const bool ym2 = y >= 2, yp2 = y + 2 < st.ny;
  const bool zm2 = z >= 2, zp2 = z + 2 < st.nz;
  const V4<T> d = ld4(diag_ptr<T>(d64, d32) + i0);
  // FP32 kernels take the coefficients the host rounded (no FP64 -> FP32
  // conversion per thread on the FP64 pipe)
  const T c1 = sizeof(T) == 4 ? (T)st.c1h : (T)st.c1;
  const T c2 = sizeof(T) == 4 ? (T)st.c2h : (T)st.c2;
  const int cb = blockIdx.y * kCpb;
  // column dots stay in registers until after the column loop, so their
  // warp sums (dependent shuffles) do not hold up the next column's loads
  T dsum[kCpb];
#pragma unroll
  for (int q = 0; q < kCpb; ++q) dsum[q] = (T)0;
#pragma unroll
  for (int q = 0; q < kCpb; ++q) {
    const int c = cb + q;
    if (c >= ncols || (DOTS && !valid)) continue;
    const T* x = X + (int64_t)c * N + i0;
    const V4<T> xc = ld4(x);
    V4<T> xlv = {{0, 0, 0, 0}}, xrv = {{0, 0, 0, 0}};
    if (xl) xlv = ld4(x - 4);
    if (xr) xrv = ld4(x + 4);
    T s1[4] = {0, 0, 0, 0}, s2[4] = {0, 0, 0, 0};
    if (ym1) { V4<T> a = ld4(x - sy); for (int k = 0; k < 4; ++k) s1[k] += a.v[k]; }
    if (yp1) { V4<T> a = ld4(x + sy); for (int k = 0; k < 4; ++k) s1[k] += a.v[k]; }
    if (zm1) { V4<T> a = ld4(x - sz); for (int k = 0; k < 4; ++k) s1[k] += a.v[k]; }
    if (zp1) { V4<T> a = ld4(x + sz); for (int k = 0; k < 4; ++k) s1[k] += a.v[k]; }
    if (R == 2) {
      if (ym2) { V4<T> a = ld4(x - 2 * sy); for (int k = 0; k < 4; ++k) s2[k] += a.v[k]; }
      if (yp2) { V4<T> a = ld4(x + 2 * sy); for (int k = 0; k < 4; ++k) s2[k] += a.v[k]; }
      if (zm2) { V4<T> a = ld4(x - 2 * sz); for (int k = 0; k < 4; ++k) s2[k] += a.v[k]; }
      if (zp2) { V4<T> a = ld4(x + 2 * sz); for (int k = 0; k < 4; ++k) s2[k] += a.v[k]; }
    }
    // x neighbours: l1/r1 at distance 1, l2/r2 at distance 2
    const T l1[4] = {xlv.v[3], xc.v[0], xc.v[1], xc.v[2]};
    const T r1[4] = {xc.v[1], xc.v[2], xc.v[3], xrv.v[0]};
    V4<T> out;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      T acc = d.v[k] * xc.v[k] + c1 * (s1[k] + l1[k] + r1[k]);
      if (R == 2) {
        const T l2 = k < 2 ? xlv.v[2 + k] : xc.v[k - 2];
        const T r2 = k > 1 ? xrv.v[k - 2] : xc.v[k + 2];
        acc += c2 * (s2[k] + l2 + r2);
      }
      out.v[k] = acc;
    }
    if (!DOTS || Y) st4(Y + (int64_t)c * N + i0, out);  // Y null: dots only
    if (DOTS)
      dsum[q] = xc.v[0] * out.v[0] + xc.v[1] * out.v[1] + xc.v[2] * out.v[2] +
                xc.v[3] * out.v[3];
  }
  if (DOTS) {
#pragma unroll
    for (int q = 0; q < kCpb; ++q) warp_dot(dsum[q], red, q);
    write_dots(red, dots, cb, ncols);
  }
}

// One point per thread, any nx (FP64).
template <typename T, int R, bool DOTS>
__global__ void __launch_bounds__(256)
    k_stencil_1(StencilOp st, int64_t N, int64_t ld, const double* __restrict__ d64,
                const float* __restrict__ d32, const T* __restrict__ X,
                T* __restrict__ Y, int ncols, double* __restrict__ dots) {
  const int64_t i0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const bool valid = i0 < N;
  if (!DOTS && !valid) return;
  const int64_t i = valid ? i0 : 0;
  __shared__ double red[kCpb][8];
  const int x = (int)(i % st.nx);
  const int64_t yz = i / st.nx;
  const int y = (int)(yz % st.ny);
  const int z = (int)(yz / st.ny);
  const int64_t sy = st.nx, sz = (int64_t)st.nx * st.ny;
  const T d = diag_ptr<T>(d64, d32)[i];
  // FP32 kernels take the coefficients the host rounded (no FP64 -> FP32
  // conversion per thread on the FP64 pipe)
  const T c1 = sizeof(T) == 4 ? (T)st.c1h : (T)st.c1;
  const T c2 = sizeof(T) == 4 ? (T)st.c2h : (T)st.c2;
  const int cb = blockIdx.y * kCpb;
  T dsum[kCpb];  // column dots, warp-summed after the column loop
#pragma unroll
  for (int q = 0; q < kCpb; ++q) dsum[q] = (T)0;
#pragma unroll
  for (int q = 0; q < kCpb; ++q) {
    const int c = cb + q;
    if (c >= ncols || (DOTS && !valid)) continue;
    const T* xp = X + (int64_t)c * ld + i;
    T s1 = 0, s2 = 0;
    if (x >= 1) s1 += xp[-1];
    if (x + 1 < st.nx) s1 += xp[1];
    if (y >= 1) s1 += xp[-sy];
    if (y + 1 < st.ny) s1 += xp[sy];
    if (z >= 1) s1 += xp[-sz];
    if (z + 1 < st.nz) s1 += xp[sz];
    T acc = d * xp[0] + c1 * s1;
    if (R == 2) {
      if (x >= 2) s2 += xp[-2];
      if (x + 2 < st.nx) s2 += xp[2];
      if (y >= 2) s2 += xp[-2 * sy];
      if (y + 2 < st.ny) s2 += xp[2 * sy];
      if (z >= 2) s2 += xp[-2 * sz];
      if (z + 2 < st.nz) s2 += xp[2 * sz];
      acc += c2 * s2;
    }
    if (!DOTS || Y) Y[(int64_t)c * ld + i] = acc;
    if (DOTS) dsum[q] = xp[0] * acc;
  }
  if (DOTS) {
#pragma unroll
    for (int q = 0; q < kCpb; ++q) warp_dot(dsum[q], red, q);
    write_dots(red, dots, cb, ncols);
  }
}

// CSR: one row per thread, KC columns at a time, so an entry's column index and
// value are read once for KC products and KC gathers are in flight together
// (one column at a time, the row cached in registers: 236 us in FP32 at
// N = 48^3, 13 entries a row, 128 columns; now 127). The last columns of a block
// that is no multiple of KC go without the others' gathers. A row's products are
// added in the order of its entries.
template <typename T>
__host__ __device__ constexpr int csr_cols() { return sizeof(T) == 4 ? 8 : 4; }

template <typename T, typename TV, bool DOTS>
__global__ void __launch_bounds__(256)
    k_csr(int64_t N, int64_t ld, const int32_t* __restrict__ rowptr,
          const int32_t* __restrict__ cols, const TV* __restrict__ vals,
          const T* __restrict__ X, T* __restrict__ Y, int ncols,
          double* __restrict__ dots) {
  constexpr int KC = csr_cols<T>();
  const int64_t r0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const bool valid = r0 < N;
  if (!DOTS && !valid) return;
  const int64_t r = valid ? r0 : 0;
  __shared__ double red[KC][8];
  const int b = valid ? rowptr[r] : 0, e = valid ? rowptr[r + 1] : 0;
  const int cb = blockIdx.y * KC, nc = min(KC, ncols - cb);
  const T* x[KC];
#pragma unroll
  for (int q = 0; q < KC; ++q) x[q] = X + (int64_t)(cb + min(q, nc - 1)) * ld;
  T acc[KC];
#pragma unroll
  for (int q = 0; q < KC; ++q) acc[q] = (T)0;
  auto row = [&](auto full) {
#pragma unroll 2
    for (int k = b; k < e; ++k) {
      const int j = cols[k];
      const T v = (T)vals[k];
#pragma unroll
      for (int q = 0; q < KC; ++q)
        if (decltype(full)::value || q < nc) acc[q] += v * __ldg(x[q] + j);
    }
  };
  if (nc == KC)
    row(std::true_type{});
  else
    row(std::false_type{});
  T d[KC];
#pragma unroll
  for (int q = 0; q < KC; ++q) {
    d[q] = (T)0;
    if (valid && q < nc) {
      if (!DOTS || Y) Y[(int64_t)(cb + q) * ld + r] = acc[q];
      if (DOTS) d[q] = x[q][r] * acc[q];
    }
  }
  if (DOTS) {
#pragma unroll
    for (int q = 0; q < KC; ++q) {
      const T t = warp_sum(d[q]);
      if ((threadIdx.x & 31) == 0) red[q][threadIdx.x >> 5] = to_f64(t);
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

// ---------------------------------------------------------------------------
// FP32 stencil with the grid planes staged in shared memory by TMA (nx % 4
// == 0, nx <= 256). A CTA owns rows y0 .. y0 + ty - 1 of one column and
// marches along z. A ring of kPlanes staged planes holds, per plane, the rows
// y0 - 2 .. y0 + ty + 1 (the halo), each loaded as one (nx x (ty + 4)) box of
// the block's 4-D tensor map (x, y, z, column); rows and planes outside the
// grid arrive as zeros, which is the Dirichlet boundary. All thirteen
// neighbours are read from shared memory, so a value comes from DRAM once
// (plus the halo rows) rather than once per neighbour through L1/L2. The z
// range is cut into grid.z chunks (each reads two halo planes on either
// side) so that about four CTAs per SM keep enough planes in flight. Thread
// (qx, ry) computes the four points x = 4 qx .. 4 qx + 3 of row y0 + ry with
// the same arithmetic, in the same order, as k_stencil_v4. With DOTS the
// column dot X_c . Y_c is accumulated in double-float per thread and the
// CTA's sum is written to dots[blockIdx.x * ncols + column].
// ---------------------------------------------------------------------------
constexpr int kPlanes = 8;
constexpr int kHalo = 2;

int plane_rows(int nx, int ny) {
  const int nxq = nx / 4;
  int ty = 256 / nxq;
  if (ty > 256 - 2 * kHalo) ty = 256 - 2 * kHalo;  // a TMA box is <= 256 high
  if (ty > ny) ty = ny;
  return ty < 1 ? 1 : ty;
}
__host__ __device__ inline int plane_stride(int nx, int ty) {
  return ((ty + 2 * kHalo) * nx + 31) & ~31;
}

template <int R, bool DOTS>
__global__ void __launch_bounds__(256)
    k_stencil_planes(const __grid_constant__ CUtensorMap map, StencilOp st,
                     const float* __restrict__ d32, float* __restrict__ Y,
                     int64_t N, int ncols, int ty, int zc,
                     double* __restrict__ dots, int* err) {
  extern __shared__ unsigned char smraw[];
  __shared__ uint64_t full[kPlanes];
  __shared__ int failed;
  __shared__ double red[8];
  const int nx = st.nx, ny = st.ny, nz = st.nz, nxq = nx >> 2;
  const int rows = ty + 2 * kHalo;
  const int pstride = plane_stride(nx, ty);
  float* planes = reinterpret_cast<float*>(
      (reinterpret_cast<uintptr_t>(smraw) + 127) & ~(uintptr_t)127);
  const int tid = threadIdx.x;
  const int y0 = blockIdx.x * ty, col = blockIdx.y;
  const int z0 = blockIdx.z * zc, z1 = min(nz, z0 + zc);
  const int qx = tid % nxq, ry = tid / nxq;
  const bool active = ry < ty && y0 + ry < ny;
  if (tid == 0) {
    for (int q = 0; q < kPlanes; ++q) tc::mbar_init(&full[q], 1);
    failed = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  const uint32_t box_bytes = (uint32_t)(rows * nx) * 4u;
  const int first = z0 - kHalo, last = z1 - 1 + kHalo;  // planes read
  int issued = first - 1;  // thread 0: last plane issued
  // plane pz goes to slot (pz - first) % kPlanes, its use number
  // (pz - first) / kPlanes giving the barrier phase
  auto slot = [&](int pz) { return (pz - first) % kPlanes; };
  auto phase = [&](int pz) { return ((pz - first) / kPlanes) & 1; };
  auto issue = [&](int pz) {
    const int q = slot(pz);
    tc::mbar_expect_tx(&full[q], box_bytes);
    tc::tma_load_4d(planes + q * pstride, &map, 0, y0 - kHalo, pz, col,
                    &full[q]);
    issued = pz;
  };
  if (tid == 0)
    for (int pz = first; pz < first + kPlanes && pz <= last; ++pz) issue(pz);
  const float c1 = st.c1h, c2 = st.c2h;  // rounded on the host
  F2 dacc = {0.f, 0.f};
  int waited = first - 1;  // last plane this thread saw land
  const int r = ry + kHalo;
  const int64_t rowoff = (int64_t)(y0 + ry) * nx + 4 * qx;
  for (int z = z0; z < z1; ++z) {
    bool ok = true;
    for (int pz = waited + 1; pz <= z + kHalo && pz <= last && ok; ++pz) {
      ok = tc::mbar_wait(&full[slot(pz)], phase(pz), err, &failed);
      if (ok) waited = pz;
    }
    if (!__syncthreads_and(ok)) break;  // the same decision in every thread
    if (active) {
      auto at = [&](int pz) {
        return planes + slot(pz) * pstride + r * nx + 4 * qx;
      };
      const float* p0 = at(z);
      const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
      const float4 xc = *reinterpret_cast<const float4*>(p0);
      const float4 xl = qx > 0 ? *reinterpret_cast<const float4*>(p0 - 4) : zero;
      const float4 xr = qx + 1 < nxq ? *reinterpret_cast<const float4*>(p0 + 4) : zero;
      const float4 ym1 = *reinterpret_cast<const float4*>(p0 - nx);
      const float4 yp1 = *reinterpret_cast<const float4*>(p0 + nx);
      const float4 zm1 = *reinterpret_cast<const float4*>(at(z - 1));
      const float4 zp1 = *reinterpret_cast<const float4*>(at(z + 1));
      const float c[4] = {xc.x, xc.y, xc.z, xc.w};
      const float a1[4] = {ym1.x, ym1.y, ym1.z, ym1.w};
      const float b1[4] = {yp1.x, yp1.y, yp1.z, yp1.w};
      const float e1[4] = {zm1.x, zm1.y, zm1.z, zm1.w};
      const float f1[4] = {zp1.x, zp1.y, zp1.z, zp1.w};
      const float l1[4] = {xl.w, xc.x, xc.y, xc.z};
      const float r1[4] = {xc.y, xc.z, xc.w, xr.x};
      float a2[4] = {0, 0, 0, 0}, b2[4] = {0, 0, 0, 0}, e2[4] = {0, 0, 0, 0},
            f2[4] = {0, 0, 0, 0};
      float l2[4] = {0, 0, 0, 0}, r2[4] = {0, 0, 0, 0};
      if (R == 2) {
        const float4 ym2 = *reinterpret_cast<const float4*>(p0 - 2 * nx);
        const float4 yp2 = *reinterpret_cast<const float4*>(p0 + 2 * nx);
        const float4 zm2 = *reinterpret_cast<const float4*>(at(z - 2));
        const float4 zp2 = *reinterpret_cast<const float4*>(at(z + 2));
        a2[0] = ym2.x; a2[1] = ym2.y; a2[2] = ym2.z; a2[3] = ym2.w;
        b2[0] = yp2.x; b2[1] = yp2.y; b2[2] = yp2.z; b2[3] = yp2.w;
        e2[0] = zm2.x; e2[1] = zm2.y; e2[2] = zm2.z; e2[3] = zm2.w;
        f2[0] = zp2.x; f2[1] = zp2.y; f2[2] = zp2.z; f2[3] = zp2.w;
        l2[0] = xl.z; l2[1] = xl.w; l2[2] = xc.x; l2[3] = xc.y;
        r2[0] = xc.z; r2[1] = xc.w; r2[2] = xr.x; r2[3] = xr.y;
      }
      const int64_t i0 = (int64_t)z * nx * ny + rowoff;
      const float4 d4 = *reinterpret_cast<const float4*>(d32 + i0);
      const float d[4] = {d4.x, d4.y, d4.z, d4.w};
      float out[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        float s1 = 0.f, s2 = 0.f;
        s1 += a1[k];
        s1 += b1[k];
        s1 += e1[k];
        s1 += f1[k];
        float acc = d[k] * c[k] + c1 * (s1 + l1[k] + r1[k]);
        if (R == 2) {
          s2 += a2[k];
          s2 += b2[k];
          s2 += e2[k];
          s2 += f2[k];
          acc += c2 * (s2 + l2[k] + r2[k]);
        }
        out[k] = acc;
      }
      if (!DOTS || Y)
        *reinterpret_cast<float4*>(Y + (int64_t)col * N + i0) =
            make_float4(out[0], out[1], out[2], out[3]);
      if (DOTS)
        dacc = df_add(dacc, F2{c[0] * out[0] + c[1] * out[1] +
                                   c[2] * out[2] + c[3] * out[3],
                               0.f});
    }
    // this thread's reads of the ring before the next TMA write there
    tc::fence_proxy_async();
    __syncthreads();
    if (tid == 0 && z - kHalo + kPlanes <= last) issue(z - kHalo + kPlanes);
  }
  // copies issued but not waited for (only after a timeout) land first
  if (tid == 0)
    for (int pz = waited + 1; pz <= issued; ++pz)
      tc::mbar_wait_own(&full[slot(pz)], phase(pz), err);
  if (DOTS) {
    // the warp sum in double-float on the FP32 pipe, one FP64 add per warp
    F2 w = dacc;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
      w = df_add(w, F2{__shfl_xor_sync(0xffffffffu, w.h, o),
                       __shfl_xor_sync(0xffffffffu, w.l, o)});
    if ((tid & 31) == 0) red[tid >> 5] = to_f64(w.h) + to_f64(w.l);
    __syncthreads();
    if (tid == 0) {
      double t = 0.0;
      for (int w = 0; w < (int)(blockDim.x + 31) / 32; ++w) t += red[w];
      dots[((size_t)blockIdx.z * gridDim.x + blockIdx.x) * ncols + col] = t;
    }
  }
}

template <int R, bool DOTS>
int launch_planes(const Operator& op, const float* X, float* Y, int ncols,
                  double* dots, cudaStream_t s) {
  const StencilOp& st = op.st;
  const int ty = plane_rows(st.nx, st.ny);
  const int tiles = ceil_div(st.ny, ty);
  // about four CTAs per SM: z chunks of at least 8 planes
  const int want = ceil_div(4 * sm_count(), tiles * ncols);
  // (and no more partial dots per column than apply_h_dots_doubles allows)
  const int cap = std::max<int>(1, (int)(ceil_div(op.N / 4, 256) / tiles));
  int chunks = std::max(1, std::min({want, ceil_div(st.nz, 8), cap}));
  const int zc = ceil_div(st.nz, chunks);
  chunks = ceil_div(st.nz, zc);
  const int threads = ((st.nx / 4) * ty + 31) & ~31;
  const size_t smem =
      (size_t)kPlanes * plane_stride(st.nx, ty) * sizeof(float) + 128;
  static std::atomic<int> attr_dev{-1};  // launches may come from several threads
  int dev = 0;
  TRM_CUDA(cudaGetDevice(&dev));
  if (attr_dev.load(std::memory_order_relaxed) != dev) {
    TRM_CUDA(cudaFuncSetAttribute(k_stencil_planes<R, DOTS>,
                                  cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  128 * 1024));
    attr_dev.store(dev, std::memory_order_relaxed);
  }
  const CUtensorMap map = tc::f32_grid_map(X, st.nx, st.ny, st.nz, ncols,
                                           ty + 2 * kHalo);
  k_stencil_planes<R, DOTS><<<dim3(tiles, ncols, chunks), threads, smem, s>>>(
      map, st, op.diag32, Y, op.N, ncols, ty, zc, dots, op.err);
  TRM_CHECK_LAUNCH();
  return tiles * chunks;  // partial dots per column
}

// The staged-plane kernel takes FP32 stencils with nx % 4 == 0 and
// nx <= 256 on 16-byte-aligned blocks.
template <typename T>
bool planes_eligible(const Operator& op, const T* X, const T* Y, int ncols) {
  if constexpr (sizeof(T) != 4) {
    return false;
  } else {
    const StencilOp& st = op.st;
    return op.kind == 0 && st.nx % 4 == 0 && st.nx <= 256 && ncols <= 65535 &&
           ((reinterpret_cast<uintptr_t>(X) | reinterpret_cast<uintptr_t>(Y) |
             reinterpret_cast<uintptr_t>(op.diag32)) & 15) == 0 &&
           plane_stride(st.nx, plane_rows(st.nx, st.ny)) * kPlanes * 4 + 128 <=
               128 * 1024 &&
           tc::encode_fn() != nullptr;
  }
}

template <typename T, bool DOTS>
int launch_vec(const Operator& op, const T* X, T* Y, int ncols, double* dots,
               cudaStream_t s);

// ---------------------------------------------------------------------------
// Register z-march (FP32): a CTA owns a tile of an x-y plane, one column and a
// chunk of z planes; a thread owns VW consecutive x points of one row (4, 2 or
// 1, as nx is a multiple of them) and walks z keeping their 2R + 1 values along
// z in registers, so per plane it reads one new value of each from DRAM and its
// x and y neighbours, which the neighbouring threads of the same tile have just
// read as their own (L1 hits), instead of four more planes through L2. There is
// no barrier inside the march, so every warp keeps its loads in flight on its
// own. With VW = 4 every point gets the same operations in the same order as in
// k_stencil_v4, else in k_stencil_1's order; with DOTS the column dot is
// accumulated in double-float per thread and the CTA's sum goes to
// dots[(blockIdx.y * gridDim.x + blockIdx.x) * ncols + column].
// Odd grids (VW = 1) took a kernel that read all twelve neighbours through L1
// and L2 for each point: 34 us at 39 x 41 x 37, 90 columns.
// ---------------------------------------------------------------------------
template <int VW>
__device__ __forceinline__ void ldv(const float* p, bool in, float (&v)[VW]) {
  if constexpr (VW == 4) {
    const float4 t = in ? __ldg(reinterpret_cast<const float4*>(p))
                        : make_float4(0.f, 0.f, 0.f, 0.f);
    v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
  } else if constexpr (VW == 2) {
    const float2 t = in ? __ldg(reinterpret_cast<const float2*>(p))
                        : make_float2(0.f, 0.f);
    v[0] = t.x; v[1] = t.y;
  } else {
    v[0] = in ? __ldg(p) : 0.f;
  }
}
template <int VW>
__device__ __forceinline__ void stv(float* p, const float (&v)[VW]) {
  if constexpr (VW == 4)
    *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
  else if constexpr (VW == 2)
    *reinterpret_cast<float2*>(p) = make_float2(v[0], v[1]);
  else
    *p = v[0];
}
// Values x0 - 2 .. x0 + VW + 1 of a row, c holding x0 .. x0 + VW - 1 and x0 a
// multiple of VW; zeros outside [0, nx).
template <int R, int VW>
__device__ __forceinline__ void row_ext(const float* p, const float (&c)[VW],
                                        int x0, int nx, float (&e)[VW + 4]) {
#pragma unroll
  for (int k = 0; k < VW; ++k) e[k + 2] = c[k];
  if constexpr (VW == 1) {
    e[1] = x0 >= 1 ? __ldg(p - 1) : 0.f;
    e[3] = x0 + 1 < nx ? __ldg(p + 1) : 0.f;
    e[0] = R == 2 && x0 >= 2 ? __ldg(p - 2) : 0.f;
    e[4] = R == 2 && x0 + 2 < nx ? __ldg(p + 2) : 0.f;
  } else {
    float a[VW], b[VW];
    ldv<VW>(p - VW, x0 >= VW, a);
    ldv<VW>(p + VW, x0 + VW < nx, b);
    e[0] = a[VW - 2];
    e[1] = a[VW - 1];
    e[VW + 2] = b[0];
    e[VW + 3] = b[1];
  }
}

template <int R, bool DOTS, int VW>
__global__ void __launch_bounds__(256, VW == 1 ? 6 : 4)
    k_stencil_zm(StencilOp st, int64_t ld, const float* __restrict__ d32,
                 const float* __restrict__ X, float* __restrict__ Y,
                 int ncols, int zc, int pack, double* __restrict__ dots) {
  __shared__ double red[8];
  const int nx = st.nx, ny = st.ny, nz = st.nz, nxq = nx / VW;
  int p, z0;  // group in the plane, first plane
  const bool active = zm_place(nxq * ny, nz, zc, pack, p, z0);
  const int x0 = active ? VW * (p % nxq) : 0, y = active ? p / nxq : 0;
  const int col = blockIdx.z;
  const int z1 = min(nz, z0 + zc);
  const int64_t sz = (int64_t)nx * ny;
  const int64_t rowoff = (int64_t)y * nx + x0;
  const float* xb = X + (int64_t)col * ld + rowoff;
  const bool ym1 = y >= 1, yp1 = y + 1 < ny, ym2 = y >= 2, yp2 = y + 2 < ny;
  const float c1 = st.c1h, c2 = st.c2h;  // rounded on the host
  // q[k]: the points in plane z - R + k (zeros outside the grid: Dirichlet);
  // q[2R + 1], plane z + R + 1, is loaded one step before it is needed so
  // that a plane's DRAM latency overlaps the arithmetic of the step before
  float q[2 * R + 2][VW];
#pragma unroll
  for (int k = 0; k < 2 * R + 1; ++k) {
    const int pz = z0 - R + k;
    ldv<VW>(xb + pz * sz, active && pz >= 0 && pz < nz, q[k]);
  }
  F2 dacc = {0.f, 0.f};
  for (int z = z0; z < z1; ++z) {
    ldv<VW>(xb + (z + R + 1) * sz, active && z + R + 1 < nz && z + 1 < z1,
            q[2 * R + 1]);
    if (active) {
      const float* pc = xb + z * sz;
      float e[VW + 4], a1[VW], b1[VW], a2[VW], b2[VW], d[VW];
      row_ext<R, VW>(pc, q[R], x0, nx, e);
      ldv<VW>(pc - nx, ym1, a1);
      ldv<VW>(pc + nx, yp1, b1);
      ldv<VW>(d32 + z * sz + rowoff, true, d);
      if (R == 2) {
        ldv<VW>(pc - 2 * nx, ym2, a2);
        ldv<VW>(pc + 2 * nx, yp2, b2);
      }
      float out[VW];
#pragma unroll
      for (int k = 0; k < VW; ++k) {
        float acc;
        if constexpr (VW == 4) {
          float s1 = 0.f, s2 = 0.f;
          s1 += a1[k];
          s1 += b1[k];
          s1 += q[R - 1][k];
          s1 += q[R + 1][k];
          acc = d[k] * q[R][k] + c1 * (s1 + e[k + 1] + e[k + 3]);
          if (R == 2) {
            s2 += a2[k];
            s2 += b2[k];
            s2 += q[0][k];
            s2 += q[2 * R][k];
            acc += c2 * (s2 + e[k] + e[k + 4]);
          }
        } else {
          // this is the FP32 stencil of such grids: x first, as in the one-point
          // kernel, and the multiply-adds written out (H C of smooth columns
          // at order 4 was 5 % further from 64 bits the other way)
          float s1 = e[k + 1] + e[k + 3];
          s1 = (s1 + a1[k]) + b1[k];
          s1 = (s1 + q[R - 1][k]) + q[R + 1][k];
          acc = fmaf(c1, s1, __fmul_rn(d[k], q[R][k]));
          if (R == 2) {
            float s2 = e[k] + e[k + 4];
            s2 = (s2 + a2[k]) + b2[k];
            s2 = (s2 + q[0][k]) + q[2 * R][k];
            acc = fmaf(c2, s2, acc);
          }
        }
        out[k] = acc;
      }
      if (!DOTS || Y) stv<VW>(Y + (int64_t)col * ld + z * sz + rowoff, out);
      if (DOTS) {
        float t = q[R][0] * out[0];
#pragma unroll
        for (int k = 1; k < VW; ++k) t += q[R][k] * out[k];
        dacc = df_add(dacc, F2{t, 0.f});
      }
    }
#pragma unroll
    for (int k = 0; k < 2 * R + 1; ++k)
#pragma unroll
      for (int u = 0; u < VW; ++u) q[k][u] = q[k + 1][u];
  }
  if (DOTS) {
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

}  // namespace

// A grid of one plane is marched along y (its rows in the planes' place).
// Launch geometry of the z-march: plane tiles of at most 256 threads (a
// multiple of 32, evened out over the tiles), z chunks so that about 3072 threads
// per SM are launched (at least four planes each; half as many leave a last
// wave, twice as many read more halo planes: 115, 112, 112 us for the
// double-float kernel at 48^3 x 128 with 2048, 3072 and 4096), and no more
// partial dots per column than apply_h_dots_doubles allows. A small plane (thin
// rods, 2-D grids with short rows) that would leave more than an eighth of its
// warps' lanes idle shares a CTA of 128 threads with other chunks.
StencilOp zm_axes(const StencilOp& st) {
  StencilOp t = st;
  if (t.nz == 1) std::swap(t.ny, t.nz);
  return t;
}
ZmShape zm_shape(const StencilOp& st, int64_t N, int ncols, int vw, int max_dots) {
  const int nq = (st.nx / vw) * st.ny;
  ZmShape z{};
  z.tiles = ceil_div(nq, 256);
  const int lanes = 32 * ceil_div(nq, 32);
  z.pack = 8 * (lanes - nq) > lanes ? std::max(1, 128 / nq) : 1;
  z.threads = 32 * ceil_div(nq * z.pack, 32 * z.tiles);
  const int per = z.pack > 1 ? nq : z.threads * z.tiles;  // threads of a chunk
  const int want =
      ceil_div((int64_t)12 * 256 * sm_count(), (int64_t)per * ncols);
  const int cap = std::max(1, max_dots / z.tiles) * z.pack;
  const int chunks = std::max(1, std::min({want, ceil_div(st.nz, 4), cap}));
  z.zc = ceil_div(st.nz, chunks);
  z.chunks = ceil_div(ceil_div(st.nz, z.zc), z.pack);
  return z;
}

namespace {

// x points per thread of the z-march for this grid and these buffers (16- and
// 8-byte vectors need the row length and the columns' spacing to match).
int zm_width(const Operator& op, const float* X, const float* Y) {
  const uintptr_t a = reinterpret_cast<uintptr_t>(X) |
                      reinterpret_cast<uintptr_t>(Y) |
                      reinterpret_cast<uintptr_t>(op.diag32);
  const int64_t n = op.st.nx | op.ld;
  if (n % 4 == 0 && a % 16 == 0) return 4;
  return n % 2 == 0 && a % 8 == 0 ? 2 : 1;
}

int max_dots_per_column(const Operator& op) {
  return (int)(apply_h_dots_doubles(op, 1));
}

template <int R, bool DOTS, int VW>
int launch_zm_v(const Operator& op, const float* X, float* Y, int ncols,
                double* dots, cudaStream_t s) {
  const StencilOp st = zm_axes(op.st);
  const ZmShape z = zm_shape(st, op.N, std::min(ncols, 65535), VW,
                             max_dots_per_column(op));
  // (the columns are the grid's last dimension: batches of what it takes)
  for (int c0 = 0; c0 < ncols; c0 += 65535) {
    const int nc = std::min(65535, ncols - c0);
    k_stencil_zm<R, DOTS, VW><<<dim3(z.tiles, z.chunks, nc), z.threads, 0, s>>>(
        st, op.ld, op.diag32, X + c0 * op.ld, Y ? Y + c0 * op.ld : nullptr,
        ncols, z.zc, z.pack, DOTS ? dots + c0 : nullptr);
    TRM_CHECK_LAUNCH();
  }
  return z.tiles * z.chunks;  // partial dots per column
}

template <bool DOTS>
int launch_zm_r(const Operator& op, const float* X, float* Y, int ncols,
                double* dots, cudaStream_t s) {
  const int vw = zm_width(op, X, Y);
  if (op.st.radius == 1)
    return vw == 4   ? launch_zm_v<1, DOTS, 4>(op, X, Y, ncols, dots, s)
           : vw == 2 ? launch_zm_v<1, DOTS, 2>(op, X, Y, ncols, dots, s)
                     : launch_zm_v<1, DOTS, 1>(op, X, Y, ncols, dots, s);
  return vw == 4   ? launch_zm_v<2, DOTS, 4>(op, X, Y, ncols, dots, s)
         : vw == 2 ? launch_zm_v<2, DOTS, 2>(op, X, Y, ncols, dots, s)
                   : launch_zm_v<2, DOTS, 1>(op, X, Y, ncols, dots, s);
}

// With nx % 4 == 0 the z-march is one of the autotuned kernels where its
// partial dots fit; on other grids it is the FP32 stencil.
template <typename T>
bool zm_eligible(const Operator& op, const T* X, const T* Y, int ncols) {
  if constexpr (sizeof(T) != 4) {
    return false;
  } else {
    if (op.kind != 0 || op.st.nx % 4 != 0 || ncols > 65535) return false;
    if (zm_width(op, X, Y) != 4) return false;
    const ZmShape z =
        zm_shape(zm_axes(op.st), op.N, ncols, 4, max_dots_per_column(op));
    return z.tiles * z.chunks <= max_dots_per_column(op);
  }
}

// Autotuned choice among the FP32 stencil kernels: the four-point kernel,
// the staged-plane kernel and the register z-march. The first apply of each
// (grid, order, columns, fused dots) in the process times every eligible
// kernel on the caller's buffers (a warm-up launch of each, then the kernels
// in turn, twice each, CUDA events on the stream) and keeps the fastest for
// the rest of the process. All compute every point with the same operations
// in the same order (the fused dots are grouped differently, so the choice
// is fixed per process: repeated solves agree bit for bit). No timing inside
// a stream capture: the four-point kernel is used there until a choice
// exists.
struct TuneKey {
  int nx, ny, nz, radius, ncols, dots;
  bool operator<(const TuneKey& o) const {
    return std::tie(nx, ny, nz, radius, ncols, dots) <
           std::tie(o.nx, o.ny, o.nz, o.radius, o.ncols, o.dots);
  }
};
std::mutex g_tune_mu;
std::map<TuneKey, int> g_tuned;  // the StencilKernel kept for a key

enum StencilKernel { kKernVec = 0, kKernPlanes = 1, kKernZm = 2 };

template <bool DOTS>
int launch_planes_r(const Operator& op, const float* X, float* Y, int ncols,
                    double* dots, cudaStream_t s) {
  return op.st.radius == 1 ? launch_planes<1, DOTS>(op, X, Y, ncols, dots, s)
                           : launch_planes<2, DOTS>(op, X, Y, ncols, dots, s);
}

template <bool DOTS>
int launch_kind(int kind, const Operator& op, const float* X, float* Y,
                int ncols, double* dots, cudaStream_t s) {
  if (kind == kKernPlanes) return launch_planes_r<DOTS>(op, X, Y, ncols, dots, s);
  if (kind == kKernZm) return launch_zm_r<DOTS>(op, X, Y, ncols, dots, s);
  return launch_vec<float, DOTS>(op, X, Y, ncols, dots, s);
}

template <bool DOTS>
int choose_kernel(const Operator& op, const float* X, float* Y, int ncols,
                  double* dots, cudaStream_t s) {
  const StencilOp& st = op.st;
  // (0: plain, 1: with dots, 2: dots only)
  const TuneKey key{st.nx, st.ny, st.nz, st.radius, ncols,
                    DOTS ? (Y ? 1 : 2) : 0};
  {
    std::lock_guard<std::mutex> lock(g_tune_mu);
    auto it = g_tuned.find(key);
    if (it != g_tuned.end()) return it->second;
  }
  int kinds[3], nk = 0;
  kinds[nk++] = kKernVec;
  if (planes_eligible(op, X, Y, ncols)) kinds[nk++] = kKernPlanes;
  if (zm_eligible(op, X, Y, ncols)) kinds[nk++] = kKernZm;
  if (nk == 1) return kKernVec;
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  TRM_CUDA(cudaStreamIsCapturing(s, &cs));
  if (cs != cudaStreamCaptureStatusNone) return kKernVec;
  constexpr int kRounds = 2;
  cudaEvent_t ev[1 + 3 * kRounds];
  for (auto& e : ev) TRM_CUDA(cudaEventCreate(&e));
  long long tuning = 0;
  capture_launches(&tuning);  // the timing launches are not the solve's
  for (int k = 0; k < nk; ++k)
    launch_kind<DOTS>(kinds[k], op, X, Y, ncols, dots, s);  // warm-up
  TRM_CUDA(cudaEventRecord(ev[0], s));
  int e = 1;
  for (int r = 0; r < kRounds; ++r)
    for (int k = 0; k < nk; ++k) {
      launch_kind<DOTS>(kinds[k], op, X, Y, ncols, dots, s);
      TRM_CUDA(cudaEventRecord(ev[e++], s));
    }
  capture_launches(nullptr);
  TRM_CUDA(cudaEventSynchronize(ev[e - 1]));
  float tot[3] = {0.f, 0.f, 0.f}, t = 0.f;
  for (int i = 1; i < e; ++i) {
    TRM_CUDA(cudaEventElapsedTime(&t, ev[i - 1], ev[i]));
    tot[(i - 1) % nk] += t;
  }
  for (auto& ee : ev) cudaEventDestroy(ee);
  int best = 0;
  for (int k = 1; k < nk; ++k)
    if (tot[k] < tot[best]) best = k;
  std::lock_guard<std::mutex> lock(g_tune_mu);
  // the first decision for a key stands (another thread may have tuned it)
  return g_tuned.emplace(key, kinds[best]).first->second;
}

template <typename T, bool DOTS>
int launch_apply(const Operator& op, const T* X, T* Y, int ncols, double* dots,
                 cudaStream_t s) {
  // one limit for every operator and type, whatever a kernel's own would be
  if (ceil_div(ncols, kCpb) > 65535)
    throw Error(-1, "too many columns for one launch");
  if constexpr (sizeof(T) == 4) {
    if (op.kind == 0 && op.st.nx % 4 != 0)
      return launch_zm_r<DOTS>(op, X, Y, ncols, dots, s);
    if (op.kind == 0 && op.st.nx % 4 == 0) {
      // TRM_STENCIL_KERNEL=vec|planes|zm overrides the tuned choice (for
      // tests and measurements; an ineligible kernel falls back to vec)
      int kind = -1;
      if (const char* f = std::getenv("TRM_STENCIL_KERNEL"))
        kind = std::strcmp(f, "planes") == 0 ? kKernPlanes
               : std::strcmp(f, "zm") == 0   ? kKernZm
                                             : kKernVec;
      // (a key's choice holds for its shape; this call's buffers must suit
      // the kernel too)
      if (kind < 0) kind = choose_kernel<DOTS>(op, X, Y, ncols, dots, s);
      if ((kind == kKernPlanes && planes_eligible(op, X, Y, ncols)) ||
          (kind == kKernZm && zm_eligible(op, X, Y, ncols)))
        return launch_kind<DOTS>(kind, op, X, Y, ncols, dots, s);
    }
  }
  return launch_vec<T, DOTS>(op, X, Y, ncols, dots, s);
}

template <typename T, bool DOTS>
int launch_vec(const Operator& op, const T* X, T* Y, int ncols, double* dots,
               cudaStream_t s) {
  const int threads = 256;
  const int gy = ceil_div(ncols, kCpb);
  dim3 grid;
  if (op.kind == 0) {
    const StencilOp& st = op.st;
    if (st.nx % 4 == 0) {
      grid = dim3(ceil_div(op.N / 4, threads), gy);
      if (st.radius == 1)
        k_stencil_v4<T, 1, DOTS><<<grid, threads, 0, s>>>(
            st, op.N, op.diag64, op.diag32, X, Y, ncols, dots);
      else
        k_stencil_v4<T, 2, DOTS><<<grid, threads, 0, s>>>(
            st, op.N, op.diag64, op.diag32, X, Y, ncols, dots);
    } else if constexpr (sizeof(T) == 8) {
      grid = dim3(ceil_div(op.N, threads), gy);
      if (st.radius == 1)
        k_stencil_1<T, 1, DOTS><<<grid, threads, 0, s>>>(
            st, op.N, op.ld, op.diag64, op.diag32, X, Y, ncols, dots);
      else
        k_stencil_1<T, 2, DOTS><<<grid, threads, 0, s>>>(
            st, op.N, op.ld, op.diag64, op.diag32, X, Y, ncols, dots);
    }
  } else {
    grid = dim3(ceil_div(op.N, threads), ceil_div(ncols, csr_cols<T>()));
    // FP32 blocks take the FP32 roundings of the values when the operator
    // holds them (the same products, no conversion per nonzero)
    if (op.csr.vals64 && (sizeof(T) == 8 || !op.csr.vals32))
      k_csr<T, double, DOTS><<<grid, threads, 0, s>>>(
          op.N, op.ld, op.csr.rowptr, op.csr.cols, op.csr.vals64, X, Y, ncols, dots);
    else
      k_csr<T, float, DOTS><<<grid, threads, 0, s>>>(
          op.N, op.ld, op.csr.rowptr, op.csr.cols, op.csr.vals32, X, Y, ncols, dots);
  }
  TRM_CHECK_LAUNCH();
  return (int)grid.x;
}

__global__ void k_stencil_diag(int64_t N, double base,
                               const double* __restrict__ V, double* d64,
                               float* d32) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N) return;
  const double d = base + (V ? V[i] : 0.0);
  d64[i] = d;
  d32[i] = (float)d;
}

template <typename TV>
__global__ void k_csr_diag(int64_t N, const int32_t* __restrict__ rowptr,
                           const int32_t* __restrict__ cols,
                           const TV* __restrict__ vals, double* d64,
                           float* d32) {
  const int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= N) return;
  double d = 0.0;
  for (int k = rowptr[r]; k < rowptr[r + 1]; ++k)
    if (cols[k] == r) d += (double)vals[k];
  d64[r] = d;
  d32[r] = (float)d;
}

// Block-wise minima of x, then the reciprocal shift.
__global__ void k_min_partial(const double* __restrict__ x, int64_t n,
                              double* out) {
  __shared__ double sm[32];
  double v = 1e300;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    v = fmin(v, x[i]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
    v = fmin(v, __shfl_xor_sync(0xffffffffu, v, o));
  if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x < 32) {
    v = threadIdx.x < (blockDim.x >> 5) ? sm[threadIdx.x] : 1e300;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
      v = fmin(v, __shfl_xor_sync(0xffffffffu, v, o));
    if (threadIdx.x == 0) out[blockIdx.x] = v;
  }
}

__global__ void k_precond(const double* __restrict__ d, int64_t n,
                          const double* __restrict__ mins, int nmins,
                          double* m64, float* m32) {
  double mn = 1e300;
  for (int k = 0; k < nmins; ++k) mn = fmin(mn, mins[k]);
  const double sigma = mn - 1.0;
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double v = 1.0 / (d[i] - sigma);
  m64[i] = v;
  m32[i] = (float)v;
}

}  // namespace

void apply_h(const Operator& op, const float* X, float* Y, int ncols,
             cudaStream_t s) {
  if (ncols > 0) launch_apply<float, false>(op, X, Y, ncols, nullptr, s);
}
void apply_h(const Operator& op, const double* X, double* Y, int ncols,
             cudaStream_t s) {
  if (ncols > 0) launch_apply<double, false>(op, X, Y, ncols, nullptr, s);
}
int apply_h_dots(const Operator& op, const float* X, float* Y, int ncols,
                 double* dots, cudaStream_t s) {
  return ncols > 0 ? launch_apply<float, true>(op, X, Y, ncols, dots, s) : 0;
}
size_t apply_h_dots_doubles(const Operator& op, int ncols) {
  const int64_t pts = (op.kind == 0 && op.st.nx % 4 == 0) ? op.N / 4 : op.N;
  return (size_t)ceil_div(pts, 256) * ncols;
}

void stencil_diag(const StencilOp&, double base, const double* V,
                  double* diag64, float* diag32, int64_t N, cudaStream_t s) {
  k_stencil_diag<<<ceil_div(N, 256), 256, 0, s>>>(N, base, V, diag64, diag32);
  TRM_CHECK_LAUNCH();
}

void csr_diag(const Operator& op, double* diag64, float* diag32,
              cudaStream_t s) {
  if (op.csr.vals64)
    k_csr_diag<double><<<ceil_div(op.N, 256), 256, 0, s>>>(
        op.N, op.csr.rowptr, op.csr.cols, op.csr.vals64, diag64, diag32);
  else
    k_csr_diag<float><<<ceil_div(op.N, 256), 256, 0, s>>>(
        op.N, op.csr.rowptr, op.csr.cols, op.csr.vals32, diag64, diag32);
  TRM_CHECK_LAUNCH();
}

void diag_preconditioner(const double* diag64, int64_t N, double* minv64,
                         float* minv32, double* work, cudaStream_t s) {
  const int nb = 256;
  k_min_partial<<<nb, 256, 0, s>>>(diag64, N, work);
  TRM_CHECK_LAUNCH();
  k_precond<<<ceil_div(N, 256), 256, 0, s>>>(diag64, N, work, nb, minv64,
                                             minv32);
  TRM_CHECK_LAUNCH();
}

}  // namespace trm
