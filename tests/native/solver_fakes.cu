// The solver's host logic (csrc/solver.cu) on the CPU: a CUDA runtime whose
// memory is host memory and whose one kernel is written out here, and block
// operations that do nothing (test_solver_host.py generates those not below). A
// timeout of a bounded device wait is the status bit that the n-th digit Gram
// leaves, as the kernel does when it gives up.
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <vector>

#include "solver.cuh"

namespace {
int g_grams = 0, g_fail_at = 0;     // digit Grams run, and which one times out
int g_copies1d = 0, g_bad_pitch = 0;
int g_clear_es = 0, g_dirty = 0;    // what G, P and HP were last cleared for
constexpr size_t kLarge = (size_t)64 << 20;  // larger requests move nothing
}  // namespace

namespace trm {
bool oz_pays(int64_t, int, int) { return true; }
void oz_gram(const OzBlock*, int, const OzBlock&, double*, double*, size_t,
             int* err, cudaStream_t) {
  if (++g_grams == g_fail_at) *err |= 2;
}
// (the list of a clear has the FP64 blocks, then G, G_prev, P and HP)
void clear_pad_rows(const PadList& l, int64_t, int64_t, int, cudaStream_t) {
  int fp64 = 0;
  while (fp64 < l.n && l.es[fp64] == 8) ++fp64;
  g_clear_es = fp64 >= 7 ? 8 : 4;
}
// the FP64 iteration's first use of H P over the padded rows
int column_dots(int64_t, int, const double*, const double*, double*,
                cudaStream_t) {
  g_dirty += g_clear_es != 8;
  return 0;
}
}  // namespace trm

// (the headers define some of these names on the host side: others are used here,
// under the runtime's link names)
extern "C" {
cudaError_t fake_cudaMallocAsync(void** p, size_t n, cudaStream_t)
    __asm__("cudaMallocAsync");
cudaError_t fake_cudaFreeAsync(void* p, cudaStream_t)
    __asm__("cudaFreeAsync");
cudaError_t fake_cudaHostAlloc(void** p, size_t n, unsigned)
    __asm__("cudaHostAlloc");
cudaError_t fake_cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t)
    __asm__("cudaMemcpyAsync");
cudaError_t fake_cudaMemcpy2DAsync(void* d, size_t dp, const void* s, size_t sp, size_t w, size_t h, cudaMemcpyKind, cudaStream_t)
    __asm__("cudaMemcpy2DAsync");
cudaError_t fake_cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t)
    __asm__("cudaMemsetAsync");
const char* fake_cudaGetErrorString(cudaError_t)
    __asm__("cudaGetErrorString");
cudaError_t fake_cudaLaunchKernel(cudaKernel_t, dim3, dim3, void** args, size_t, cudaStream_t)
    __asm__("__cudaLaunchKernel");

cudaError_t fake_cudaMallocAsync(void** p, size_t n, cudaStream_t) {
  *p = std::calloc(1, n);
  return *p ? cudaSuccess : cudaErrorMemoryAllocation;
}
cudaError_t fake_cudaFreeAsync(void* p, cudaStream_t) {
  std::free(p);
  return cudaSuccess;
}
cudaError_t fake_cudaHostAlloc(void** p, size_t n, unsigned) {
  *p = std::calloc(1, n);
  return cudaSuccess;
}
cudaError_t fake_cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind,
                                 cudaStream_t) {
  if (n >= kLarge) ++g_copies1d;
  else std::memcpy(d, s, n);
  return cudaSuccess;
}
// (the runtime takes pitches up to 2^31 - 1 bytes)
cudaError_t fake_cudaMemcpy2DAsync(void* d, size_t dp, const void* s, size_t sp,
                              size_t w, size_t h, cudaMemcpyKind, cudaStream_t) {
  if (dp > 0x7FFFFFFF || sp > 0x7FFFFFFF) {
    ++g_bad_pitch;
    return cudaErrorInvalidPitchValue;
  }
  for (size_t r = 0; r < h; ++r)
    std::memcpy((char*)d + r * dp, (const char*)s + r * sp, w);
  return cudaSuccess;
}
cudaError_t fake_cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t) {
  if (n < kLarge) std::memset(p, v, n);
  return cudaSuccess;
}
const char* fake_cudaGetErrorString(cudaError_t) { return "fake"; }
// k_set_restart(IterScalars*, int keep), the only kernel of solver.cu
cudaError_t fake_cudaLaunchKernel(cudaKernel_t, dim3, dim3, void** args, size_t,
                               cudaStream_t) {
  auto* sc = *static_cast<trm::IterScalars**>(args[0]);
  sc->restart = 1;
  sc->status &= *static_cast<int*>(args[1]);
  return cudaSuccess;
}
}

static trm_options options(int precision) {
  trm_options o{};
  o.precision = precision;
  o.max_iter = 100;
  o.lag = 2;
  o.graphs = 1;
  o.switch_tol[0] = 1e-5;
  return o;
}

// status of a solve whose n-th digit Gram times out, then of one without
static int solve_status(trm::Solver& s, int n) {
  g_grams = 0;
  g_fail_at = n;
  double lam[8], eg;
  const int st = s.solve(lam, &eg, nullptr, 0, nullptr, nullptr);
  g_fail_at = 0;
  return st;
}
static int ritz_status(trm::Solver& s, int n) {
  g_grams = 0;
  g_fail_at = n;
  static double C[64 * 8], lam[8], res[8];
  int st = TRM_OK;
  try {
    s.rayleigh_ritz(C, lam, res);
  } catch (const trm::Error& e) {
    st = e.status;
  }
  g_fail_at = 0;
  return st;
}

static int timeouts() {
  int bad = 0;
  for (int precision : {TRM_FP64, TRM_MP2, TRM_MIXED}) {
    trm::Solver s(64, 8, 1e-10, options(precision));
    s.init_stencil(4, 4, 4, 2, 1.0, nullptr);
    bad += solve_status(s, 0) != TRM_OK;
    const int grams = g_grams;
    for (int n = 1; n <= grams; ++n) {
      const int st = solve_status(s, n), after = solve_status(s, 0);
      std::printf("precision %d gram %d of %d: %d, then %d\n", precision, n,
                  grams, st, after);
      bad += st != TRM_ETIMEOUT || after != TRM_OK;
    }
    bad += ritz_status(s, 0) != TRM_OK || g_grams < 2;
    for (int n = g_grams; n >= 1; --n) {
      const int st = ritz_status(s, n), after = ritz_status(s, 0);
      std::printf("precision %d ritz gram %d: %d, then %d\n", precision, n, st,
                  after);
      bad += st != TRM_ETIMEOUT || after != TRM_OK;
    }
  }
  return bad;
}

// A block from and to the host whose columns are 2^31 bytes and more apart
// (N % 4 != 0: the solver's own are padded).
static int large_columns() {
  const int64_t N = ((int64_t)1 << 28) + 1;
  trm::Solver s(N, 2, 1e-10, options(TRM_FP64));
  s.init_stencil((int)N, 1, 1, 2, 1.0, nullptr);
  g_copies1d = 0;
  double lam[2], eg, C[2];  // (the fake moves nothing of this size)
  const int st = s.solve(lam, &eg, C, 0, C, nullptr);
  std::printf("large columns: %d, %d copies, %d refused\n", st, g_copies1d,
              g_bad_pitch);
  return st != TRM_OK || g_copies1d != 4 || g_bad_pitch != 0;
}

// The generalized mixed ladder on padded columns: full SP with FP32 blocks in
// G, P and HP, then FP64 ones in the same places.
static int generalized_padding() {
  const int n = 5, N = n * n * n;
  std::vector<int> rp(N + 1), ci(N);
  std::vector<double> v(N, 1.0);
  for (int i = 0; i < N; ++i) {
    ci[i] = i;
    rp[i + 1] = i + 1;
  }
  trm::Solver s(N, 8, 1e-10, options(TRM_MIXED));
  s.init_stencil(n, n, n, 2, 1.0, nullptr);
  s.init_overlap(rp.data(), ci.data(), v.data());
  const int st = solve_status(s, 0);
  std::printf("generalized: %d, %d digit Grams, %d on uncleared padding\n", st,
              g_grams, g_dirty);
  return st != TRM_OK || g_grams < 6 || g_dirty != 0;
}

int main(int argc, char** argv) {
  const char* what = argc > 1 ? argv[1] : "";
  try {
    if (!std::strcmp(what, "timeouts")) return timeouts() != 0;
    if (!std::strcmp(what, "large_columns")) return large_columns();
    if (!std::strcmp(what, "generalized")) return generalized_padding();
  } catch (const std::exception& e) {
    std::printf("%s: %s\n", what, e.what());
    return 1;
  }
  return 2;
}
