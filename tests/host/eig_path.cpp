// Host logic of the truncated SVD's eigensolver path, without a GPU: api.cu
// compiled by the host compiler, the CUDA runtime and the kernel families it calls
// replaced by the stand-ins below.  Prints one line per scenario; the test
// (tests/test_eig_path_host.py) holds the expected lines.
#include <cstdlib>

#include "api.cu"

// ---- stand-ins

static int g_reduces = 0;                                  // calls of eig_reduce
static int g_fail_at = 0;                                  // the call that fails (1 = the first), 0 = none
static cudaError_t g_fail_with = cudaErrorMemoryAllocation;
static double g_residual = 0;                              // what norm2_scale reports of the residual
static int g_status = 0;                                   // status of the next truncations
static float (*g_lam)(int) = nullptr;                      // the spectrum eig_spectrum reports

extern "C" {
cudaError_t cudaMalloc(void** p, size_t n) { *p = std::calloc(1, n ? n : 1); return *p ? cudaSuccess : cudaErrorMemoryAllocation; }
cudaError_t cudaFree(void* p) { std::free(p); return cudaSuccess; }
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) { std::memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) { std::memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) { std::memset(d, v, n); return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }     // the launch that failed has already read and cleared it
const char* cudaGetErrorString(cudaError_t) { return "stand-in error"; }
}

namespace dmrgc {
size_t eig_work_bytes(int n, int kk) { return (size_t)16 * n * (kk + 8); }
size_t trunc_bytes(int n) { return sizeof(TruncResult) + 12 * (size_t)n; }
cudaError_t gemm_simt(const GemmArgs&, bool, cudaStream_t) { return cudaSuccess; }
cudaError_t gemm_tc(const GemmArgs&, int, TcWork&, int*, cudaStream_t, int*) { return cudaSuccess; }
void TcWork::release() {}
cudaError_t eig_reduce(void*, int, int, void*, cudaStream_t, int*) {
  return ++g_reduces == g_fail_at ? g_fail_with : cudaSuccess;
}
cudaError_t eig_spectrum(const void*, int, int kk, float* lam, EigHead* head, cudaStream_t) {
  for (int i = 0; i < kk; ++i) lam[i] = g_lam(i);
  head->err = 0;
  head->unit = 1.0;
  head->trace = 2.0;
  return cudaSuccess;
}
cudaError_t eig_select(const void*, int, int, int most, double cut, double, double, void*, void* res, void*, int,
                       cudaStream_t, int*) {
  TruncResult t{};
  t.status = g_status;
  if (g_lam)
    while (t.k < most && g_lam(t.k) > cut * cut * g_lam(0)) ++t.k;
  else
    t.k = most;
  std::memcpy(res, &t, sizeof(t));
  return cudaSuccess;
}
cudaError_t norm2_scale(void*, long long, bool, double* out, double*, bool, cudaStream_t) { *out = g_residual; return cudaSuccess; }
cudaError_t place_columns(const void*, int, int, void*, int, int, int, cudaStream_t) { return cudaSuccess; }
}  // namespace dmrgc

// ---- scenarios

static void setup(dmrgc_ctx& c, int chi, int bonds) {
  c.opt = dmrgc_options{};
  c.opt.precision = DMRGC_TF32X3;
  c.fp64 = false;
  c.esz = 8;
  c.N = bonds;
  c.chi = chi;
  c.sweep_cut = 2e-5;
  c.zero_rel = 1e-5;
  c.tie_rel = 1e-5;
  c.eig_declined.assign(bonds, 0);
  g_reduces = 0;
  g_fail_at = 0;
  g_status = 0;
  g_residual = 0;
  g_lam = [](int i) { return (float)std::pow(10.0, -0.03 * i); };
}

// a theta of rows x cols, updated left to right (right = false) or right to left
static dmrgc_status visit(dmrgc_ctx& c, int bond, int rows, int cols, bool right, bool& done) {
  static std::vector<char> theta;
  theta.resize((size_t)8 * rows * cols);
  DevBuf out;
  int k = 0;
  const dmrgc_status s = eig_try(&c, bond, theta.data(), right ? cols : rows, right ? rows : cols, right, c.sweep_cut, 0.0,
                                 out, right ? 2 : 0, k, done, true);
  cudaFree(out.p);
  return s;
}

static void failed_reduction() {
  for (int rows : {250, 400})          // one Gram matrix only; in stages
    for (int at = 1; at <= (rows > 256 ? 2 : 1); ++at)
      for (cudaError_t e : {cudaErrorMemoryAllocation, cudaErrorLaunchOutOfResources, cudaErrorInvalidConfiguration}) {
        dmrgc_ctx c;
        setup(c, 200, 4);
        g_fail_at = at;
        g_fail_with = e;
        g_residual = 1e-3;             // the first stage leaves something: a second one follows
        bool done = false;
        const dmrgc_status s = visit(c, 0, rows, rows, false, done);
        std::printf("reduce rows=%d call=%d error=%d: status=%d done=%d declined=%lld\n", rows, at, (int)e, (int)s, (int)done,
                    (long long)c.stats.eig_fallbacks);
      }
}

// One update at bond 1: prints what became of it.
static void update(dmrgc_ctx& c, const char* name, int rows, int cols, bool right) {
  const long long skipped = c.stats.eig_skipped, declined = c.stats.eig_fallbacks;
  const int reduces = g_reduces;
  bool done = false;
  const dmrgc_status s = visit(c, 1, rows, cols, right, done);
  note_resolvable(&c, 1);
  const char* what = s != DMRGC_OK ? "error" : done ? "taken" : c.stats.eig_skipped > skipped ? "skipped"
                     : c.stats.eig_fallbacks > declined ? "declined" : g_reduces > reduces ? "lost" : "not tried";
  std::printf("%s %d x %d %s: %s\n", name, rows, cols, right ? "right to left" : "left to right", what);
}

static void visits() {
  dmrgc_ctx a;
  setup(a, 600, 4);   // every row may be kept; the residual is noise
  update(a, "tall then wide", 600, 250, false);
  update(a, "tall then wide", 600, 250, true);
  update(a, "tall then wide", 600, 250, false);
  dmrgc_ctx b;
  setup(b, 600, 4);
  g_residual = 1e-3;  // what 250 rows decline, 300 rows take in stages
  update(b, "grown bond", 250, 400, false);
  update(b, "grown bond", 250, 400, false);
  update(b, "grown bond", 300, 400, false);
  update(b, "grown bond", 250, 400, false);
  dmrgc_ctx d;
  setup(d, 200, 4);
  g_status = 1;       // unresolved by one Gram matrix
  update(d, "one Gram matrix", 250, 400, false);
  update(d, "one Gram matrix", 250, 400, false);
  g_status = 0;
  update(d, "one Gram matrix", 400, 400, true);
  dmrgc_ctx e;
  setup(e, 200, 4);
  g_status = 1;       // not taken in stages either: nothing takes it
  update(e, "stages", 400, 400, false);
  g_status = 0;
  update(e, "stages", 400, 400, true);
  update(e, "stages", 250, 400, false);
  dmrgc_ctx l;
  setup(l, 200, 4);   // rank below chi: the sweep's cut sets the count, a wider one is resolved
  update(l, "low rank", 250, 150, false);
  update(l, "low rank", 250, 200, false);
  l.sweep_cut = 4e-3;
  update(l, "low rank, wide cut", 250, 150, false);
  dmrgc_ctx r;
  setup(r, 200, 4);
  r.opt.log_rank_records = 1;   // the recorded spectrum decides
  g_status = 1;
  r.last_tr.tail = 1.0;
  update(r, "records", 400, 400, false);
  g_status = 0;
  r.last_tr.by_cut = 0;
  r.last_tr.tail = 1.0;
  note_resolvable(&r, 1);       // a Jacobi SVD found it resolved
  update(r, "records", 400, 400, true);
}

int main(int argc, char** argv) {
  (void)argc;
  if (std::string(argv[1]) == "failed_reduction") failed_reduction();
  if (std::string(argv[1]) == "visits") visits();
  return 0;
}
