// Batched complex GEMM on CUDA cores (FFMA / DFMA), any operand op.
//
// This is the FP64 path's contraction engine and the FP32 reference path of
// the complex64 modes.  One CTA of 256 threads computes a 64x64 tile of C;
// every thread owns a 4x4 block of complex accumulators.  Operand tiles are
// staged in shared memory with the loads ordered along the operand's
// contiguous index so that global reads coalesce for every op.
//
// Small products use 16 x 16 tiles instead, one output per thread, with K
// split over the CTAs of a cluster (gemm_small_kernel): GB300's FP64 rate is two
// FMAs per SM and clock, so one 64 x 64 tile of a product with K = 64 keeps a
// single SM busy for a quarter of a millisecond while the others idle.
#include "common.cuh"

#include <algorithm>
#include <climits>

namespace dmrgc {
namespace {

constexpr int BM = 64, BN = 64, TM = 4, TN = 4, NT = 256;

template <typename R> struct Tile;
template <> struct Tile<float> { static constexpr int BK = 16; };
template <> struct Tile<double> { static constexpr int BK = 8; };

template <typename R, int BK>
__global__ void __launch_bounds__(NT) gemm_kernel(GemmArgs g) {
  using C2 = typename cplx<R>::T;
  __shared__ C2 As[BK][BM + 1];
  __shared__ C2 Bs[BK][BN + 1];

  const int bz = blockIdx.z;
  const int i1 = bz / g.b2, i2 = bz % g.b2;
  const C2* __restrict__ A = reinterpret_cast<const C2*>(g.A) + i1 * g.sA1 + i2 * g.sA2;
  const C2* __restrict__ B = reinterpret_cast<const C2*>(g.B) + i1 * g.sB1 + i2 * g.sB2;
  C2* __restrict__ C = reinterpret_cast<C2*>(g.C) + i1 * g.sC1 + i2 * g.sC2;
  const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
  const int tid = threadIdx.x;
  const int tx = tid % (BN / TN), ty = tid / (BN / TN);

  C2 acc[TM][TN];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) acc[i][j] = C2{0, 0};

  const bool a_kfast = (g.opA == OP_N || g.opA == OP_R);
  const bool a_conj = (g.opA == OP_C || g.opA == OP_R);
  const bool b_nfast = (g.opB == OP_N || g.opB == OP_R);
  const bool b_conj = (g.opB == OP_C || g.opB == OP_R);

  for (int k0 = 0; k0 < g.K; k0 += BK) {
    // A tile: BM x BK
    for (int e = tid; e < BM * BK; e += NT) {
      int mm, kk;
      if (a_kfast) { kk = e % BK; mm = e / BK; } else { mm = e % BM; kk = e / BM; }
      const int m = m0 + mm, k = k0 + kk;
      C2 v{0, 0};
      if (m < g.M && k < g.K) {
        v = a_kfast ? A[(long long)m * g.lda + k] : A[(long long)k * g.lda + m];
        if (a_conj) v.y = -v.y;
      }
      As[kk][mm] = v;
    }
    // B tile: BK x BN
    for (int e = tid; e < BN * BK; e += NT) {
      int nn, kk;
      if (b_nfast) { nn = e % BN; kk = e / BN; } else { kk = e % BK; nn = e / BK; }
      const int n = n0 + nn, k = k0 + kk;
      C2 v{0, 0};
      if (n < g.N && k < g.K) {
        v = b_nfast ? B[(long long)k * g.ldb + n] : B[(long long)n * g.ldb + k];
        if (b_conj) v.y = -v.y;
      }
      Bs[kk][nn] = v;
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < BK; ++kk) {
      C2 a[TM], b[TN];
#pragma unroll
      for (int i = 0; i < TM; ++i) a[i] = As[kk][ty + i * (BM / TM)];
#pragma unroll
      for (int j = 0; j < TN; ++j) b[j] = Bs[kk][tx + j * (BN / TN)];
#pragma unroll
      for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) {
          acc[i][j].x = fma(a[i].x, b[j].x, acc[i][j].x);
          acc[i][j].x = fma(-a[i].y, b[j].y, acc[i][j].x);
          acc[i][j].y = fma(a[i].x, b[j].y, acc[i][j].y);
          acc[i][j].y = fma(a[i].y, b[j].x, acc[i][j].y);
        }
    }
    __syncthreads();
  }
  const R ar = (R)g.alpha_re, ai = (R)g.alpha_im;
#pragma unroll
  for (int i = 0; i < TM; ++i) {
    const int m = m0 + ty + i * (BM / TM);
    if (m >= g.M) continue;
#pragma unroll
    for (int j = 0; j < TN; ++j) {
      const int n = n0 + tx + j * (BN / TN);
      if (n >= g.N) continue;
      C2 v{acc[i][j].x * ar - acc[i][j].y * ai, acc[i][j].x * ai + acc[i][j].y * ar};
      C2* dst = C + (long long)m * g.ldc + n;
      if (g.beta_one) { C2 o = *dst; v.x += o.x; v.y += o.y; }
      *dst = v;
    }
  }
}

// 16 x 16 tile per cluster of S CTAs (gridDim.x = N tiles x S): CTA ks sums the
// K blocks ks, ks + S, .. of 16, the partial tiles meet in shared memory and each
// CTA adds its share of the outputs over the cluster in the order of the ranks,
// so every product is reproducible.  At this rate the operand traffic (512 bytes
// per 1024 FMAs) and the shared-memory loads hide behind the FMAs.  The products
// of the 12-qubit FP64 run (M, N <= 128, K <= 1024) averaged 142 us on 64 x 64
// tiles; with these the whole run went from 117 to 45 ms, the single-site
// step at 4 x 5, chi = 24 from 159 to 52 ms.
constexpr int ST = 16;

__device__ __forceinline__ unsigned gs_map(unsigned addr, unsigned rank) {
  unsigned r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ double2 gs_load(unsigned addr, double2) {
  double2 v;
  asm volatile("ld.shared::cluster.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ float2 gs_load(unsigned addr, float2) {
  float2 v;
  asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ void gs_cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

template <typename R>
__global__ void __launch_bounds__(ST * ST) gemm_small_kernel(GemmArgs g, int S) {
  using C2 = typename cplx<R>::T;
  __shared__ __align__(16) C2 As[2][ST][ST + 1];
  __shared__ __align__(16) C2 Bs[2][ST][ST + 1];
  __shared__ __align__(16) C2 part[ST * ST];
  const int bz = blockIdx.z;
  const int i1 = bz / g.b2, i2 = bz % g.b2;
  const C2* __restrict__ A = reinterpret_cast<const C2*>(g.A) + i1 * g.sA1 + i2 * g.sA2;
  const C2* __restrict__ B = reinterpret_cast<const C2*>(g.B) + i1 * g.sB1 + i2 * g.sB2;
  C2* __restrict__ C = reinterpret_cast<C2*>(g.C) + i1 * g.sC1 + i2 * g.sC2;
  const int ks = blockIdx.x % S;
  const int m0 = blockIdx.y * ST, n0 = (int)(blockIdx.x / S) * ST;
  const int tid = threadIdx.x, lo = tid % ST, hi = tid / ST;
  const bool a_kfast = (g.opA == OP_N || g.opA == OP_R), a_conj = (g.opA == OP_C || g.opA == OP_R);
  const bool b_nfast = (g.opB == OP_N || g.opB == OP_R), b_conj = (g.opB == OP_C || g.opB == OP_R);
  // this thread's operand elements: the fast index of the source runs over lo
  const int am = m0 + (a_kfast ? hi : lo), ak = a_kfast ? lo : hi;
  const int bn = n0 + (b_nfast ? lo : hi), bk = b_nfast ? hi : lo;
  auto load_a = [&](int k0) {
    C2 v{0, 0};
    const int k = k0 + ak;
    if (am < g.M && k < g.K) v = a_kfast ? A[(long long)am * g.lda + k] : A[(long long)k * g.lda + am];
    if (a_conj) v.y = -v.y;
    return v;
  };
  auto load_b = [&](int k0) {
    C2 v{0, 0};
    const int k = k0 + bk;
    if (bn < g.N && k < g.K) v = b_nfast ? B[(long long)k * g.ldb + bn] : B[(long long)bn * g.ldb + k];
    if (b_conj) v.y = -v.y;
    return v;
  };
  C2 acc{0, 0};
  const int step = ST * S;
  C2 ra = load_a(ks * ST), rb = load_b(ks * ST);
  int buf = 0;
  for (int k0 = ks * ST; k0 < g.K; k0 += step) {
    As[buf][ak][am - m0] = ra;
    Bs[buf][bk][bn - n0] = rb;
    __syncthreads();
    if (k0 + step < g.K) {   // the next block's loads run under this block's FMAs
      ra = load_a(k0 + step);
      rb = load_b(k0 + step);
    }
#pragma unroll
    for (int kk = 0; kk < ST; ++kk) {
      const C2 a = As[buf][kk][hi], b = Bs[buf][kk][lo];
      acc.x = fma(a.x, b.x, acc.x);
      acc.x = fma(-a.y, b.y, acc.x);
      acc.y = fma(a.x, b.y, acc.y);
      acc.y = fma(a.y, b.x, acc.y);
    }
    buf ^= 1;   // the next block goes to the other buffer: no second barrier
  }
  const R ar = (R)g.alpha_re, ai = (R)g.alpha_im;
  auto store = [&](int e, C2 v) {
    const int m = m0 + e / ST, n = n0 + e % ST;
    if (m >= g.M || n >= g.N) return;
    C2 o{v.x * ar - v.y * ai, v.x * ai + v.y * ar};
    C2* dst = C + (long long)m * g.ldc + n;
    if (g.beta_one) { const C2 c = *dst; o.x += c.x; o.y += c.y; }
    *dst = o;
  };
  if (S == 1) {
    store(tid, acc);
    return;
  }
  part[tid] = acc;
  __syncwarp();
  gs_cluster_sync();
  const int share = ST * ST / S;   // S divides 256
  if (tid < share) {
    const int e = ks * share + tid;
    const unsigned mine = (unsigned)__cvta_generic_to_shared(&part[e]);
    C2 sum{0, 0};
    for (int r = 0; r < S; ++r) {
      const C2 v = gs_load(gs_map(mine, r), C2{});
      sum.x += v.x;
      sum.y += v.y;
    }
    store(e, sum);
  }
  __syncwarp();
  gs_cluster_sync();   // every partial has been read before a CTA leaves
}

int simt_sms() {
  int dev = 0, n = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
  return n > 0 ? n : 148;
}

// Split of a small-tile product on `sms` SMs (0: use the 64 x 64 tiles): the fewest
// waves of tiles over the SMs times the K blocks of one tile (at least 2 K blocks per
// CTA, clusters of at most 8 CTAs), if that is less than what the 64 x 64 tiles
// cost in the same unit, with 10% for the larger tile's lower overhead per FMA.
//
// FP64: both kernels run at the FMA rate once their SMs are busy, so a large tile
// costs 16 small ones.
// FP32: the small kernel issues two shared-memory loads for four FMAs and reaches
// half of the large one's rate, which in turn needs several CTAs an SM: w waves of
// large tiles cost 7 + 6 w (fitted to 41 sizes).  1024 x 1024 x 512: 139 us on large
// tiles, 207 on small ones; 2048 x 1024 x 512: 233 and 406; 512 x 512 x 512: 107 and
// 62; 64 x 64 x 512: 106 and 8; even at 160 large tiles.  A split has to save a
// sixteenth here (640 x 1024 x 512: 135 us in one piece, 151 in eight).
int small_split(const GemmArgs& g, long long batch, bool fp64, long long sms) {
  const long long t64 = (long long)((g.M + BM - 1) / BM) * ((g.N + BN - 1) / BN) * batch;
  const long long tm = (g.M + ST - 1) / ST, tn = (g.N + ST - 1) / ST;
  if (tm > 65535 || tn * 8 > INT_MAX) return 0;
  const long long kb = std::max<long long>(1, (g.K + ST - 1) / ST);
  const long long waves = (t64 + sms - 1) / sms;
  const long long c64 = (fp64 ? waves * (BM * BN / (ST * ST)) : 7 + 6 * waves) * kb;
  long long best = LLONG_MAX;
  int split = 1;
  for (int s = 1; s <= 8 && (s == 1 || kb >= 2 * s); s *= 2) {
    const long long c = (tm * tn * batch * s + sms - 1) / sms * ((kb + s - 1) / s);
    if (fp64 || s == 1 ? c < best : 16 * c < 15 * best) { best = c; split = s; }
  }
  return 10 * best < 9 * c64 ? split : 0;
}

template <typename R>
cudaError_t launch_small(const GemmArgs& g, long long batch, int S, cudaStream_t st) {
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = S;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.gridDim = dim3((unsigned)((g.N + ST - 1) / ST * S), (unsigned)((g.M + ST - 1) / ST), (unsigned)batch);
  cfg.blockDim = dim3(ST * ST);
  cfg.stream = st;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, gemm_small_kernel<R>, g, S);
}

}  // namespace

cudaError_t gemm_simt(const GemmArgs& g, bool fp64, cudaStream_t st) {
  if (g.M <= 0 || g.N <= 0 || g.b1 <= 0 || g.b2 <= 0) return cudaSuccess;
  const long long batch = (long long)g.b1 * g.b2;
  if (batch > 65535) return cudaErrorInvalidConfiguration;
  const long long gy = (g.M + BM - 1) / BM;
  if (gy > 65535) return cudaErrorInvalidConfiguration;
  dim3 grid((g.N + BN - 1) / BN, (unsigned)gy, (unsigned)batch);
  // an empty contraction (K <= 0) writes C = 0, or leaves it with beta
  if (const int S = small_split(g, batch, fp64, simt_sms())) return fp64 ? launch_small<double>(g, batch, S, st) : launch_small<float>(g, batch, S, st);
  if (fp64)
    gemm_kernel<double, Tile<double>::BK><<<grid, NT, 0, st>>>(g);
  else
    gemm_kernel<float, Tile<float>::BK><<<grid, NT, 0, st>>>(g);
  return cudaGetLastError();
}

}  // namespace dmrgc
