// Fixed-rank approximation of the density matrix (Sec. 3.2).
//
// rho = L L^dagger with L a 2^n x m factor stored column-major (column c is a
// state vector at offset c * 2^n).  A channel with Kraus operators E_1..E_K
// (Eq. 3) produces L' = [E_1 L | ... | E_K L] (M = K m columns); the best
// rank-r approximation of L' L'^dagger is L' W_r, where W_r holds the r
// leading eigenvectors of the M x M Gram matrix G = L'^dagger L'.
//
// One-qubit and diagonal channels take three kernels: the FP64 moments of L
// that G is made of (k_moments), the eigensolver (k_eig_truncate: a one-block FP32
// Jacobi refined to FP64, with the canonical basis rule for tied eigenvalues),
// and the projection L <- scale * L' W_r straight from L (k_project_fused).  Dense
// two-qubit channels and explicit truncations go through L': Kraus expansion,
// Gram matrix in FP64 (block partials plus a fixed-order sum), the same
// eigensolver, and the projection from L'.
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <type_traits>

#include "internal.cuh"

namespace qs {

namespace {

constexpr int kExpBlock = 256;
constexpr int kGramRows = 64;            // rows of L' per shared-memory tile of the Gram kernel
constexpr int kGramTarget = 512;         // about this many row blocks per member (fixed by n)
constexpr int kTriMax = kMaxGramDim * (kMaxGramDim + 1) / 2;
constexpr int kJacobiSweeps = 40;        // bound on the eigensolver's sweeps
constexpr double kTieTol = 1e-10;        // cluster: within 1e-10 * Lambda_1
constexpr double kGsAccept = 1e-3;       // residual norm to accept a projection
constexpr double kGsFallback = 1e-8;
constexpr double kRotTol = 4e-16;        // rotate while |a_pq| > kRotTol * max|a_ii|
constexpr int kJacobiSweeps32 = 12;      // bound on the FP32 pre-pass

__device__ __forceinline__ uint64_t insert0(uint64_t v, int s) {
  return ((v >> s) << (s + 1)) | (v & ((1ull << s) - 1));
}

// Entry (row, col) of operator `op` of the xi-averaged Kraus set of a noisy
// gate U (Eqs. 5-6 and 8-9) at noise level e: rotation noise -> U N with N
// the tensor product over the targets (target 0 the low local bit) of
// sqrt(l1) I or sqrt(l2) J, J = [[0, 1], [-1, 0]], l1,2 = (1 +- e^{-2e^2})/2;
// phase noise -> U diag(1, .., 1, sqrt P) and U diag(0, .., 0, sqrt(1 - P)),
// P = e^{-e^2}.
__device__ double2 kraus_entry(const KrausGate& g, double e, int op, int row, int col) {
  const int D = 1 << g.k;
  double nre[4];                                         // column `col` of N (real)
  if (g.noise == QS_NOISE_ROTATION) {
    const double q = exp(-2.0 * e * e);
    const double s1 = sqrt(0.5 * (1.0 + q)), s2 = sqrt(0.5 * (1.0 - q));
    for (int x = 0; x < D; ++x) {
      double v = 1.0;
      for (int j = 0; j < g.k; ++j) {
        const int w = (op >> j) & 1, rb = (x >> j) & 1, cb = (col >> j) & 1;
        v *= w == 0 ? (rb == cb ? s1 : 0.0) : (rb == 0 && cb == 1 ? s2 : (rb == 1 && cb == 0 ? -s2 : 0.0));
      }
      nre[x] = v;
    }
  } else {
    const double P = exp(-e * e);
    for (int x = 0; x < D; ++x) nre[x] = 0.0;
    if (op == 0) nre[col] = col == D - 1 ? sqrt(P) : 1.0;
    else if (col == D - 1) nre[col] = sqrt(1.0 - P);
  }
  double re = 0.0, im = 0.0;                             // (U N)[row][col]
  for (int x = 0; x < D; ++x) {
    re += g.U[2 * (row * D + x)] * nre[x];
    im += g.U[2 * (row * D + x) + 1] * nre[x];
  }
  return make_double2(re, im);
}

// Lp_b[a m_b + c] = E_a L_b[c] for member b = blockIdx.y; one thread per
// (group, column) of a two-qubit channel.  The Kraus operators are E, or the gate's
// at the member's noise level.  Block (0, b) records M_b = K m_b.  REAL: L and the
// E_a are real (imaginary parts zero), real arithmetic.
template <typename R, bool REAL>
__global__ void __launch_bounds__(kExpBlock) k_kraus_expand(const cplx<R>* __restrict__ L,
                                                            cplx<R>* __restrict__ Lp, int n, int rcap, int mcap,
                                                            Targets tg, const double* __restrict__ E, int K,
                                                            RankCounts rc, const KrausGate g) {
  using C = cplx<R>;
  constexpr int D = 4;
  __shared__ C sE[8 * D * D];
  const int b = blockIdx.y;
  if (g.k > 0) {
    // the member's averaged Kraus set, built here from its noise level
    const double e = g.e_member ? g.e_member[b] : (g.e_run ? *g.e_run : g.e_value);
    for (int i = threadIdx.x; i < K * D * D; i += blockDim.x) {
      const double2 v = kraus_entry(g, e, i / (D * D), (i / D) % D, i % D);
      sE[i] = mk<R>((R)v.x, (R)v.y);
    }
  } else {
    for (int i = threadIdx.x; i < K * D * D; i += blockDim.x) sE[i] = mk<R>((R)E[2 * i], (R)E[2 * i + 1]);
  }
  const int m = rc.cols[b];
  if (blockIdx.x == 0 && threadIdx.x == 0) rc.M[b] = K * m;
  __syncthreads();
  const uint64_t N = 1ull << n;
  const uint64_t groups = N >> 2;
  const uint64_t total = groups * (uint64_t)m;
  const C* Lb = L + (uint64_t)b * rcap * N;
  C* Lpb = Lp + (uint64_t)b * mcap * N;
  for (uint64_t w = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; w < total;
       w += (uint64_t)gridDim.x * blockDim.x) {
    const int c = (int)(w / groups);
    const uint64_t g = w - (uint64_t)c * groups;
    uint64_t base = g;
#pragma unroll
    for (int j = 0; j < 2; ++j) base = insert0(base, tg.sorted[j]);
    if constexpr (REAL) {
      R v[D];
#pragma unroll
      for (int l = 0; l < D; ++l) v[l] = Lb[(uint64_t)c * N + base + tg.off[l]].x;
      for (int a = 0; a < K; ++a) {
        C* out = Lpb + (uint64_t)(a * m + c) * N + base;
#pragma unroll
        for (int r = 0; r < D; ++r) {
          R acc = R(0);
#pragma unroll
          for (int q = 0; q < D; ++q) acc = fma(sE[(a * D + r) * D + q].x, v[q], acc);
          out[tg.off[r]] = mk<R>(acc, R(0));
        }
      }
    } else {
      C v[D];
#pragma unroll
      for (int l = 0; l < D; ++l) v[l] = Lb[(uint64_t)c * N + base + tg.off[l]];
      for (int a = 0; a < K; ++a) {
        C* out = Lpb + (uint64_t)(a * m + c) * N + base;
#pragma unroll
        for (int r = 0; r < D; ++r) {
          C acc = mk<R>(R(0), R(0));
#pragma unroll
          for (int q = 0; q < D; ++q) acc = cfma(sE[(a * D + r) * D + q], v[q], acc);
          out[tg.off[r]] = acc;
        }
      }
    }
  }
}

// (p, q), p <= q, of entry idx of the upper triangle of an M x M matrix,
// row-major (row p starts at p M - p (p - 1) / 2)
__device__ __forceinline__ void tri_pq(int idx, int M, int* p, int* q) {
  const float h = (float)M + 0.5f;
  int pp = (int)(h - sqrtf(fmaxf(h * h - 2.f * (float)idx, 0.f)));
  if (pp * M - pp * (pp - 1) / 2 > idx) --pp;            // the square root's rounding
  else if ((pp + 1) * M - (pp + 1) * pp / 2 <= idx) ++pp;
  *p = pp;
  *q = pp + idx - (pp * M - pp * (pp - 1) / 2);
}

// Gram partials of member b = blockIdx.y: block x sums rows
// [x rows_per_block, (x + 1) rows_per_block) of L'_b, in tiles of kGramRows
// rows through shared memory, for every entry (p <= q) of the upper triangle
// (each entry a fixed-order FP64 sum).  Blocks of 16 tiles of rows or more
// (n >= 19) run kGramThreads threads, smaller ones half as many (their
// channels are latency-bound, and fewer warps meet at each barrier).  A thread
// owns entries idx, idx + blockDim, ...; when the block is large and the
// triangle has at most blockDim / 2 entries (M <= 21 at 512 threads) its rows
// are split instead among G = min(blockDim / tri, kGramRows) groups of
// threads (group g takes the tile rows x = g mod G), so nearly every thread
// works and the FP64 units of all four schedulers are busy, and the groups'
// sums are added in group order at the end.  Partial layout
// [member][block][kTriMax] complex.  The row split and the block size depend
// only on n, so a member's result does not depend on the batch.
constexpr int kGramThreads = 512;

template <typename R, bool REAL>
__global__ void __launch_bounds__(kGramThreads) k_gram_partials(const cplx<R>* __restrict__ Lp, int n, int mcap,
                                                                int rows_per_block, RankCounts rc,
                                                                double* __restrict__ partials) {
  using T = typename std::conditional<REAL, double, double2>::type;
  // threads: kGramThreads where rows are split (blocks of 16 tiles or more), else half
  constexpr int kOwn = (kTriMax + kGramThreads / 2 - 1) / (kGramThreads / 2);
  const int nt = (int)blockDim.x;
  __shared__ T tile[kMaxGramDim][kGramRows + 1];
  __shared__ double2 gsum[kGramThreads];
  const int b = blockIdx.y;
  const int M = rc.M[b];
  const int tri = M * (M + 1) / 2;
  // row groups per entry (at most one per row of a tile); only where a block
  // has rows enough to keep them busy (from n = 19 on), the small factors'
  // channels being latency-bound
  const int G = tri <= nt / 2 && rows_per_block >= 16 * kGramRows ? min(nt / tri, kGramRows) : 1;
  const int g = G > 1 ? (int)threadIdx.x / tri : 0;    // this thread's group (G: idle)
  const uint64_t N = 1ull << n;
  const cplx<R>* Lpb = Lp + (uint64_t)b * mcap * N;
  int ep[kOwn], eq[kOwn];
  double re[kOwn], im[kOwn], re2[kOwn];
#pragma unroll
  for (int j = 0; j < kOwn; ++j) {
    const int idx = G > 1 ? (j == 0 ? (int)threadIdx.x % tri : tri) : (int)threadIdx.x + nt * j;
    ep[j] = eq[j] = 0;
    if (idx < tri && g < G) tri_pq(idx, M, &ep[j], &eq[j]);
    re[j] = im[j] = re2[j] = 0.0;
  }
  const uint64_t r0 = (uint64_t)blockIdx.x * rows_per_block;
  for (int s = 0; s < rows_per_block; s += kGramRows) {
    __syncthreads();
    for (int i = threadIdx.x; i < M * kGramRows; i += blockDim.x) {
      const int p = i / kGramRows, x = i % kGramRows;
      const uint64_t row = r0 + s + x;
      const cplx<R> a = row < N ? Lpb[(uint64_t)p * N + row] : mk<R>(R(0), R(0));
      if constexpr (REAL) tile[p][x] = a.x;
      else tile[p][x] = make_double2(a.x, a.y);
    }
    __syncthreads();
    if (G > 1) {
      if (g >= G) continue;
      const int p = ep[0], q = eq[0];
      if constexpr (REAL) {
        int k = 0;
        for (int x = g; x < kGramRows; x += G, ++k) {
          if (k & 1) re2[0] = fma(tile[p][x], tile[q][x], re2[0]);
          else re[0] = fma(tile[p][x], tile[q][x], re[0]);
        }
      } else {
        for (int x = g; x < kGramRows; x += G) {
          const double2 a = tile[p][x], c = tile[q][x];
          re[0] = fma(a.x, c.x, fma(a.y, c.y, re[0]));   // conj(a) * c, four FMAs
          im[0] = fma(a.x, c.y, fma(-a.y, c.x, im[0]));
        }
      }
      continue;
    }
#pragma unroll
    for (int j = 0; j < kOwn; ++j) {
      if ((int)threadIdx.x + nt * j >= tri) continue;
      const int p = ep[j], q = eq[j];
      if constexpr (REAL) {
        for (int x = 0; x < kGramRows; x += 2) {
          re[j] = fma(tile[p][x], tile[q][x], re[j]);
          re2[j] = fma(tile[p][x + 1], tile[q][x + 1], re2[j]);
        }
      } else {
        for (int x = 0; x < kGramRows; ++x) {
          const double2 a = tile[p][x], c = tile[q][x];
          re[j] = fma(a.x, c.x, fma(a.y, c.y, re[j]));   // conj(a) * c, four FMAs
          im[j] = fma(a.x, c.y, fma(-a.y, c.x, im[j]));
        }
      }
    }
  }
  double* out = partials + ((size_t)b * gridDim.x + blockIdx.x) * 2 * kTriMax;
  if (G > 1) {
    // the groups' sums of each entry, added in group order
    if (g < G) gsum[threadIdx.x] = make_double2(re[0] + re2[0], im[0]);
    __syncthreads();
    if ((int)threadIdx.x < tri) {
      double sr = 0.0, si = 0.0;
      for (int k = 0; k < G; ++k) {
        sr += gsum[k * tri + threadIdx.x].x;
        si += gsum[k * tri + threadIdx.x].y;
      }
      out[2 * threadIdx.x] = sr;
      out[2 * threadIdx.x + 1] = si;
    }
    return;
  }
#pragma unroll
  for (int j = 0; j < kOwn; ++j) {
    const int idx = (int)threadIdx.x + nt * j;
    if (idx >= tri) continue;
    out[2 * idx] = re[j] + re2[j];
    out[2 * idx + 1] = im[j];
  }
}

// G_b[p][q] = the sum over member b's partial blocks (fixed-order tree), one
// block per entry of the upper triangle (grid.x) and member (grid.y); the
// lower triangle by conjugation.
__global__ void __launch_bounds__(256) k_gram_reduce(const double* __restrict__ partials, int blocks,
                                                     RankCounts rc, double* __restrict__ small, int sstride) {
  const int b = blockIdx.y, idx = blockIdx.x;
  const int M = rc.M[b];
  if (idx >= M * (M + 1) / 2) return;                    // the whole block
  int p, q;
  tri_pq(idx, M, &p, &q);
  __shared__ double sre[256], sim[256];
  double re = 0.0, im = 0.0;
  const double* part = partials + (size_t)b * blocks * 2 * kTriMax;
  for (int k = threadIdx.x; k < blocks; k += blockDim.x) {
    re += part[(size_t)k * 2 * kTriMax + 2 * idx];
    im += part[(size_t)k * 2 * kTriMax + 2 * idx + 1];
  }
  sre[threadIdx.x] = re;
  sim[threadIdx.x] = im;
  __syncthreads();
  for (int o = 128; o; o >>= 1) {
    if ((int)threadIdx.x < o) {
      sre[threadIdx.x] += sre[threadIdx.x + o];
      sim[threadIdx.x] += sim[threadIdx.x + o];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    double* G = small + (size_t)b * sstride + kSmallG;
    G[2 * (p * M + q)] = sre[0];
    G[2 * (p * M + q) + 1] = p == q ? 0.0 : sim[0];
    G[2 * (q * M + p)] = sre[0];
    G[2 * (q * M + p) + 1] = p == q ? 0.0 : -sim[0];
  }
}

__device__ __forceinline__ double2 zmul(double2 a, double2 b) {
  return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__device__ __forceinline__ double2 zconj(double2 a) { return make_double2(a.x, -a.y); }
__device__ __forceinline__ double2 zadd(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }

// Scalar helpers for the real (double) and complex (double2) Jacobi variants.
__device__ __forceinline__ double tmul(double a, double b) { return a * b; }
__device__ __forceinline__ double2 tmul(double2 a, double2 b) { return zmul(a, b); }
__device__ __forceinline__ double tadd(double a, double b) { return a + b; }
__device__ __forceinline__ double2 tadd(double2 a, double2 b) { return zadd(a, b); }
__device__ __forceinline__ double tconj(double a) { return a; }
__device__ __forceinline__ double2 tconj(double2 a) { return zconj(a); }
__device__ __forceinline__ double tre(double a) { return a; }
__device__ __forceinline__ double tre(double2 a) { return a.x; }
__device__ __forceinline__ double tabs2(double a) { return a * a; }
__device__ __forceinline__ double tabs2(double2 a) { return a.x * a.x + a.y * a.y; }
template <typename T> __device__ __forceinline__ T tscal(double v);
template <> __device__ __forceinline__ double tscal<double>(double v) { return v; }
template <> __device__ __forceinline__ double2 tscal<double2>(double v) { return make_double2(v, 0.0); }
__device__ __forceinline__ double tscale(double a, double v) { return a * v; }
__device__ __forceinline__ double2 tscale(double2 a, double v) { return make_double2(a.x * v, a.y * v); }
// the same for the FP32 pre-pass (float / float2)
__device__ __forceinline__ float tmul(float a, float b) { return a * b; }
__device__ __forceinline__ float2 tmul(float2 a, float2 b) { return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x); }
__device__ __forceinline__ float tadd(float a, float b) { return a + b; }
__device__ __forceinline__ float2 tadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float tconj(float a) { return a; }
__device__ __forceinline__ float2 tconj(float2 a) { return make_float2(a.x, -a.y); }
__device__ __forceinline__ float tre(float a) { return a; }
__device__ __forceinline__ float tre(float2 a) { return a.x; }
__device__ __forceinline__ float tabs2(float a) { return a * a; }
__device__ __forceinline__ float tabs2(float2 a) { return a.x * a.x + a.y * a.y; }
template <> __device__ __forceinline__ float tscal<float>(double v) { return (float)v; }
template <> __device__ __forceinline__ float2 tscal<float2>(double v) { return make_float2((float)v, 0.f); }
__device__ __forceinline__ float tscale(float a, float v) { return a * v; }
__device__ __forceinline__ float2 tscale(float2 a, float v) { return make_float2(a.x * v, a.y * v); }
// e^{-i arg a} for a != 0: the sign of a real a, conj(a) / |a| for a complex
// one (FP64 unit modulus: an FP32 reciprocal square root refined by two
// Newton steps in FP64)
__device__ __forceinline__ double unit_phase(double a) { return a < 0.0 ? -1.0 : 1.0; }
__device__ __forceinline__ double2 unit_phase(double2 a) {
  const double a2 = a.x * a.x + a.y * a.y;
  double y = (double)rsqrtf((float)a2);
  y = y * fma(-0.5 * a2 * y, y, 1.5);
  y = y * fma(-0.5 * a2 * y, y, 1.5);
  return make_double2(a.x * y, -a.y * y);
}
__device__ __forceinline__ float unit_phase(float a) { return a < 0.f ? -1.f : 1.f; }
__device__ __forceinline__ float2 unit_phase(float2 a) {
  const float inv = rsqrtf(a.x * a.x + a.y * a.y);
  return make_float2(a.x * inv, -a.y * inv);
}

// conversions between the FP64 and FP32 forms
__device__ __forceinline__ float to32f(float a) { return a; }
__device__ __forceinline__ float2 to32f(float2 a) { return a; }
__device__ __forceinline__ float to32f(double a) { return (float)a; }
__device__ __forceinline__ float2 to32f(double2 a) { return make_float2((float)a.x, (float)a.y); }
__device__ __forceinline__ float to32(double a) { return (float)a; }
__device__ __forceinline__ float2 to32(double2 a) { return make_float2((float)a.x, (float)a.y); }
__device__ __forceinline__ double to64(float a) { return a; }
__device__ __forceinline__ double2 to64(float2 a) { return make_double2(a.x, a.y); }


template <typename T> __device__ __forceinline__ T tscal_d();        // zero
template <> __device__ __forceinline__ double tscal_d<double>() { return 0.0; }
template <> __device__ __forceinline__ double2 tscal_d<double2>() { return make_double2(0.0, 0.0); }
template <typename T> __device__ __forceinline__ T gsm(double2 v);    // an entry of G
template <> __device__ __forceinline__ double gsm<double>(double2 v) { return v.x; }
template <> __device__ __forceinline__ double2 gsm<double2>(double2 v) { return v; }

// ---------------------------------------------------------------------------
// One-qubit and diagonal channels without L' (every noisy Hadamard, every
// phase-noise gate, T1/T2 relaxation).  With E_a the Kraus operators and l_j
// the rows of L whose target bits have the local value j,
//   G_(a,p),(b,q) = sum_ij (E_a^dagger E_b)_ij T_ij,pq,   T_ij,pq = sum over groups conj(l_i,p) l_j,q,
// so the Gram matrix needs only the moments T of the m columns of L, and
//   L'[i] W = sum_j l_j V_ij,   V_ij = sum_a (E_a)_ij W_a,
// so the projection reads L and writes L.  L' (K m columns) is neither
// written nor read, and the FP64 work of the Gram matrix falls from
// K m (K m + 1) / 2 multiply-adds a row to (2 m^2 + m) / 2 (dense one-qubit
// operators) or m (m + 1) / 2 (diagonal ones: T_ll only), that of the projection
// of a diagonal channel from K m keep to m keep.

constexpr int kMomThreads = 256;
constexpr int kMomLanes = 8;             // threads that share an entry (they take every 8th group of rows)
constexpr int kMomSlots = kMomThreads / kMomLanes;
constexpr int kMomOwn = 5;               // entries of T per thread and pass over the rows
constexpr int kMomChunk = kMomSlots * kMomOwn;
constexpr int kMomTile = 1024;           // elements of L in a shared-memory tile
constexpr int kMomBlocks = 304;          // row blocks per member at most: two per SM
constexpr int kMomGroup = 16;            // row blocks whose sums the last of them adds
constexpr int kMomGroups = (kMomBlocks + kMomGroup - 1) / kMomGroup;
constexpr int kMomUnit = 32;             // groups of rows: the granularity of the split
static_assert(kMomUnit % kMomLanes == 0 && kMomChunk <= kMomThreads, "moment tiling");

// entries of T for m columns: dense (D = 2): T_00, T_11 (upper triangles), T_01
// (all); diagonal: T_ll, l < D (upper triangles)
__host__ __device__ constexpr int mom_entries(int m, int D, bool diag) {
  return diag ? D * (m * (m + 1) / 2) : m * (m + 1) + m * m;
}
// (i, p, j, q) of entry e, as tile rows i m + p and j m + q
__device__ __forceinline__ void mom_entry(int e, int m, bool diag, int* a, int* b) {
  const int tri = m * (m + 1) / 2;
  if (!diag && e >= 2 * tri) {
    const int k = e - 2 * tri;
    *a = k / m;
    *b = m + k % m;
    return;
  }
  const int l = e / tri;
  int p, q;
  tri_pq(e % tri, m, &p, &q);
  *a = l * m + p;
  *b = l * m + q;
}
// Row blocks of a member and groups of rows per block: a function of n and D
// alone, so a member's sums do not depend on the batch.
struct MomSplit { int blocks; uint64_t per; };
// doubles of one row of partial sums: the most entries any form has at this rank
__host__ __device__ inline int mom_stride(int rank) {
  const int a = mom_entries(rank, 2, false), b = mom_entries(rank, 4, true);
  return 2 * (a > b ? a : b);
}
__host__ __device__ inline MomSplit mom_split(int n, int kq) {
  const uint64_t units = ((1ull << n) >> kq) / kMomUnit > 0 ? ((1ull << n) >> kq) / kMomUnit : 1;
  const uint64_t per = (units + kMomBlocks - 1) / kMomBlocks;
  return {(int)((units + per - 1) / per), per * kMomUnit};
}

// Moments of member b = blockIdx.y over the groups of row block blockIdx.x.
// Bound by the FP64 pipe (a warp's FP64 instruction holds its scheduler for 64
// cycles), so nearly every lane carries a useful multiply-add: eight threads
// share up to kMomOwn entries at a time and take every eighth group of a tile of
// rows in shared memory, and the next tile's elements are in registers meanwhile.
// More than kMomChunk entries (m > 8) take several passes over the rows.  The
// eight sums of an entry meet in shared memory (32 threads an entry would cost 31
// FP64 additions there, as much as a quarter of the products at 15 qubits; blocks
// of 512 threads, one per SM, left the pipe idle between their phases: five jobs
// of ranks 1..8 at 15 qubits 54 us, 43 as it is; the Gram matrix of L' took 99 and
// its reduction 11, after 20 to write L').  The last block of every kMomGroup adds the
// group's sums in block order, so the eigensolver's block has kMomGroups values
// per entry left to add, not one per row block (its single SM would need 5 us
// and more for those).
// Block (0, b) also writes member b's Kraus operators for the eigensolver, off
// its critical path.
template <typename R, bool REAL, int KQ, bool DIAG>
__global__ void __launch_bounds__(kMomThreads) k_moments(const cplx<R>* __restrict__ L, int n, int rcap, Targets tg, int K,
                                                         RankCounts rc, double* __restrict__ partials, int estride,
                                                         uint32_t* __restrict__ counters, double* __restrict__ small,
                                                         int sstride, const __grid_constant__ KrausGate gate) {
  using T = typename std::conditional<REAL, double, double2>::type;
  constexpr int D = 1 << KQ, W = REAL ? 1 : 2;
  constexpr int kLoad = kMomTile / kMomThreads;
  constexpr size_t kTileBytes = (kMomTile + D * kMaxRank) * sizeof(T);
  constexpr size_t kRedBytes = (size_t)kMomChunk * (kMomLanes + 1) * sizeof(double);
  __shared__ __align__(16) unsigned char raw[kTileBytes > kRedBytes ? kTileBytes : kRedBytes];
  __shared__ uint32_t last_of_group;
  T* tile = reinterpret_cast<T*>(raw);
  double* red = reinterpret_cast<double*>(raw);
  const int b = blockIdx.y, lane = threadIdx.x % kMomLanes, slot = threadIdx.x / kMomLanes;
  const int m = rc.cols[b];
  if (blockIdx.x == 0 && threadIdx.x == 0) rc.M[b] = K * m;
  if (blockIdx.x == 0 && gate.k > 0) {
    const double e = gate.e_member ? gate.e_member[b] : (gate.e_run ? *gate.e_run : gate.e_value);
    double2* E = reinterpret_cast<double2*>(small + (size_t)b * sstride + kSmallE);
    for (int i = threadIdx.x; i < K * D * D; i += kMomThreads) E[i] = kraus_entry(gate, e, i / (D * D), (i / D) % D, i % D);
  }
  const int ne = mom_entries(m, D, DIAG);
  const uint64_t N = 1ull << n, groups = N >> KQ;
  const MomSplit sp = mom_split(n, KQ);
  const uint64_t g0 = (uint64_t)blockIdx.x * sp.per;
  const uint64_t g1 = g0 + sp.per < groups ? g0 + sp.per : groups;
  // groups per tile: whole warps' worth, at most kMomTile elements
  const int dm = D * m;
  const int XG = max(1, min(kMomTile / dm, 256) / kMomLanes) * kMomLanes;
  const int pitch = XG + 1;
  const int elems = dm * XG;
  const cplx<R>* Lb = L + (uint64_t)b * rcap * N;
  T next[kLoad];
  auto fetch = [&](uint64_t gt) {
#pragma unroll
    for (int i = 0; i < kLoad; ++i) {
      const int el = threadIdx.x + i * kMomThreads;
      T v = tscal_d<T>();
      if (el < elems) {
        const int jp = el / XG, x = el - jp * XG;
        const int j = jp / m, p = jp - j * m;
        const uint64_t g = gt + x;
        if (g < g1) {
          uint64_t row = g;
#pragma unroll
          for (int k = 0; k < KQ; ++k) row = insert0(row, tg.sorted[k]);
          const cplx<R> a = Lb[(uint64_t)p * N + row + tg.off[j]];
          if constexpr (REAL) v = a.x;
          else v = make_double2(a.x, a.y);
        }
      }
      next[i] = v;
    }
  };
  // a member's partial sums: one row per row block, then one per group of them
  const int gcount = ((int)gridDim.x + kMomGroup - 1) / kMomGroup;
  double* mine = partials + (size_t)b * (gridDim.x + gcount) * estride;
  double* out = mine + (size_t)blockIdx.x * estride;
  for (int e0 = 0; e0 < ne; e0 += kMomChunk) {
    int ra[kMomOwn], rb[kMomOwn];
    double re[kMomOwn], im[kMomOwn];
#pragma unroll
    for (int k = 0; k < kMomOwn; ++k) {
      const int e = e0 + slot + k * kMomSlots;
      int a = 0, c = 0;
      if (e < ne) mom_entry(e, m, DIAG, &a, &c);
      ra[k] = a * pitch;
      rb[k] = c * pitch;
      re[k] = im[k] = 0.0;
    }
    fetch(g0);
    for (uint64_t gt = g0; gt < g1; gt += XG) {
      __syncthreads();
#pragma unroll
      for (int i = 0; i < kLoad; ++i) {
        const int el = threadIdx.x + i * kMomThreads;
        if (el < elems) { const int jp = el / XG; tile[jp * pitch + (el - jp * XG)] = next[i]; }
      }
      __syncthreads();
      if (gt + XG < g1) fetch(gt + XG);
      const int xn = (int)(g1 - gt < (uint64_t)XG ? g1 - gt : (uint64_t)XG);
      for (int x = lane; x < xn; x += kMomLanes) {
#pragma unroll
        for (int k = 0; k < kMomOwn; ++k) {
          if (e0 + slot + k * kMomSlots >= ne) break;
          const T a = tile[ra[k] + x], c = tile[rb[k] + x];
          if constexpr (REAL) {
            re[k] = fma(a, c, re[k]);
          } else {
            re[k] = fma(a.x, c.x, fma(a.y, c.y, re[k]));   // conj(a) c
            im[k] = fma(a.x, c.y, fma(-a.y, c.x, im[k]));
          }
        }
      }
    }
    // the eight sums of each entry, in lane order
#pragma unroll
    for (int part = 0; part < W; ++part) {
      __syncthreads();
#pragma unroll
      for (int k = 0; k < kMomOwn; ++k) red[(slot + k * kMomSlots) * (kMomLanes + 1) + lane] = part ? im[k] : re[k];
      __syncthreads();
      const int e = (int)threadIdx.x;
      if (e < kMomChunk && e0 + e < ne) {
        double s[2] = {};
#pragma unroll
        for (int k = 0; k < kMomLanes; ++k) s[k & 1] += red[e * (kMomLanes + 1) + k];
        out[(size_t)W * (e0 + e) + part] = s[0] + s[1];
      }
    }
    __syncthreads();
  }
  // the last block of a group of row blocks adds the group's sums
  const int grp = blockIdx.x / kMomGroup;
  const int first = grp * kMomGroup, count = min(kMomGroup, (int)gridDim.x - first);
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last_of_group = atomicInc(&counters[b * kMomGroups + grp], (uint32_t)count - 1) == (uint32_t)count - 1;
  __syncthreads();
  if (!last_of_group) return;
  __threadfence();
  const double* src = mine + (size_t)first * estride;
  double* dst = mine + ((size_t)gridDim.x + grp) * estride;
  for (int i = threadIdx.x; i < ne * W; i += kMomThreads) {
    double v[kMomGroup];
#pragma unroll
    for (int k = 0; k < kMomGroup; ++k) v[k] = k < count ? __ldcg(src + (size_t)k * estride + i) : 0.0;
    double s = 0.0;
#pragma unroll
    for (int k = 0; k < kMomGroup; ++k) s += v[k];
    dst[i] = s;
  }
}

// L_b[i][c] = sum_j sum_p l_j,p V_ij[p][c] for c < keep_b, in place; columns
// keep_b.. of the old m_b cleared, then m_b = keep_b.  V (the scale folded in)
// comes from the eigensolver's block.  One thread per row and run of CB
// columns; a block holds whole groups, and all of it has read before any of it
// writes.  FP64-pipe bound: D m keep (dense) or m keep (diagonal) multiply-adds
// a row; a thread per row and column run rather than per group, and small blocks
// (one per 128 / runs rows, no grid stride) share the FP64 work out over the SMs:
// with 256 threads and two blocks of a rank-8 member on some SMs, one on others,
// the pipe was busy 100 % on the first and 51 % on average.  Five jobs of ranks
// 1..8 at 15 qubits, one-qubit channel: 37 us, 105 from L' (which has K m columns).
constexpr int kProjThreads = 128;
template <typename R, bool REAL, int KQ, bool DIAG, int CB>
__global__ void __launch_bounds__(kProjThreads) k_project_fused(cplx<R>* __restrict__ L, int n, int rcap, Targets tg, int K,
                                                                int nrun, const double* __restrict__ small, int sstride,
                                                                RankCounts rc) {
  using T = typename std::conditional<REAL, double, double2>::type;
  constexpr int D = 1 << KQ;
  constexpr int NV = DIAG ? D : D * D;
  extern __shared__ __align__(16) unsigned char proj_sm[];
  T* sV = reinterpret_cast<T*>(proj_sm);                 // [ij][p][c], c padded to nrun CB
  const int b = blockIdx.y;
  const int keep = rc.keep[b], m = rc.M[b] / K;
  const int cw = nrun * CB;
  const double* V = small + (size_t)b * sstride + kSmallV;
  for (int i = threadIdx.x; i < NV * m * cw; i += kProjThreads) {
    const int c = i % cw, r = i / cw;
    T v = tscal_d<T>();
    if (c < keep) {
      if constexpr (REAL) v = V[r * keep + c];
      else v = make_double2(V[2 * (r * keep + c)], V[2 * (r * keep + c) + 1]);
    }
    sV[i] = v;
  }
  __syncthreads();
  if (blockIdx.x == 0 && threadIdx.x == 0) rc.cols[b] = keep;
  const uint64_t N = 1ull << n;
  cplx<R>* Lb = L + (uint64_t)b * rcap * N;
  const int rows = kProjThreads / nrun;                  // rows of a block, whole groups
  const int run = threadIdx.x / rows, rl = threadIdx.x % rows;
  const int per = rows >> KQ;                            // groups of a block
  const int i = rl / per;                                // local row index of the thread
  const int c0 = run * CB, nc = keep - c0;
  for (uint64_t gb = (uint64_t)blockIdx.x * per; gb < (N >> KQ); gb += (uint64_t)gridDim.x * per) {
    const uint64_t g = gb + rl % per;
    const bool live = run < nrun && g < (N >> KQ);
    uint64_t base = g;
#pragma unroll
    for (int k = 0; k < KQ; ++k) base = insert0(base, tg.sorted[k]);
    T acc[CB];
#pragma unroll
    for (int c = 0; c < CB; ++c) acc[c] = tscal_d<T>();
    if (live && c0 < keep) {
#pragma unroll
      for (int j = 0; j < (DIAG ? 1 : D); ++j) {
        const int jr = DIAG ? i : j;
        const cplx<R>* col = Lb + base + tg.off[jr];
        const T* v = sV + (size_t)(DIAG ? i : i * D + j) * m * cw + c0;
#pragma unroll 4
        for (int p = 0; p < m; ++p, col += N, v += cw) {
          const cplx<R> a = *col;
#pragma unroll
          for (int c = 0; c < CB; ++c) {
            if (c >= nc) break;                          // the same across the warps of a run
            const T w = v[c];
            if constexpr (REAL) {
              acc[c] = fma((double)a.x, w, acc[c]);
            } else {
              const double ax = a.x, ay = a.y;
              acc[c].x = fma(ax, w.x, fma(-ay, w.y, acc[c].x));
              acc[c].y = fma(ax, w.y, fma(ay, w.x, acc[c].y));
            }
          }
        }
      }
    }
    __syncthreads();                                     // whole groups have been read
    if (live) {
      cplx<R>* o = Lb + base + tg.off[i];
#pragma unroll
      for (int c = 0; c < CB; ++c) {
        if (c0 + c < keep) {
          if constexpr (REAL) o[(uint64_t)(c0 + c) * N] = mk<R>((R)acc[c], R(0));
          else o[(uint64_t)(c0 + c) * N] = mk<R>((R)acc[c].x, (R)acc[c].y);
        }
      }
      if (run == 0)
        for (int c = keep; c < m; ++c) o[(uint64_t)c * N] = mk<R>(R(0), R(0));
    }
  }
}
constexpr int kJP = kMaxGramDim + 1;                    // pitch of the eigensolver's arrays
constexpr int kEigThreads = 256;                        // two warps per scheduler

// ---------------------------------------------------------------------------
// Parallel cyclic Jacobi on the Hermitian (or real symmetric) A (M x M, pitch
// kJP), accumulating V (V <- V R, from a unitary start).  Each step applies Mp / 2
// disjoint rotations of the round-robin schedule: pair 0 = (Mp - 1, s), pair i =
// ((s + i) mod (Mp - 1), (s - i) mod (Mp - 1)).  T is float / float2, where most of
// the work is done (a warp's FP64 instruction holds its scheduler for about 64
// cycles on this GPU), or double / double2, for matrices refine() declines, from a
// basis in which A is nearly diagonal.
//
// A step is a chain of latencies: every warp tests the step's pairs (and all go
// on to the next step when none rotates), warp 0 finds the rotations (lane =
// pair: a phase makes a_pq real, then the classical angle; in FP64 the tangent is
// found in FP32 -- any tangent gives an exactly unitary rotation, the next sweep
// removes what is left -- and cos, sin and the phase are refined by Newton steps),
// the first warps update A, the others V, in place.  Of A only the 2 x 2 blocks
// (rows of pair i, columns of pair j >= i) are computed, one of their two columns
// a thread, and written below the diagonal as conjugates; what no rotating pair
// touches is skipped.
//
// FP32: a pair rotates while |a_pq| > tol sqrt(a_pp a_qq) (G is a Gram matrix:
// its small eigenvalues are graded, and the refinement needs their vectors as
// well separated as the large ones') and above kFloor32 of the largest
// diagonal entry; a sweep whose tangents were all below 2e-4 ends the loop, what
// it leaves is below their square.  FP64: while |a_pq| > tol * max |a_ii|; the
// loop ends with a sweep without rotations.  Returns false if the sweep bound was
// reached.
constexpr float kFloor32 = 1e-13f;
template <typename T> struct Rot {
  decltype(tre(T{})) c, s;               // R = [[c, s], [-s ph, c ph]]
  T sp, cp;                              // s ph, c ph
};

__device__ __forceinline__ float cmacc(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ float2 cmacc(float2 a, float2 b, float2 c) {
  return make_float2(fmaf(a.x, b.x, fmaf(-a.y, b.y, c.x)), fmaf(a.x, b.y, fmaf(a.y, b.x, c.y)));
}
__device__ __forceinline__ double cmacc(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ double2 cmacc(double2 a, double2 b, double2 c) {
  return make_double2(fma(a.x, b.x, fma(-a.y, b.y, c.x)), fma(a.x, b.y, fma(a.y, b.x, c.y)));
}
// real factor: c + v a
__device__ __forceinline__ float rmacc(float v, float a, float c) { return fmaf(v, a, c); }
__device__ __forceinline__ float2 rmacc(float v, float2 a, float2 c) { return make_float2(fmaf(v, a.x, c.x), fmaf(v, a.y, c.y)); }
__device__ __forceinline__ double rmacc(double v, double a, double c) { return fma(v, a, c); }
__device__ __forceinline__ double2 rmacc(double v, double2 a, double2 c) { return make_double2(fma(v, a.x, c.x), fma(v, a.y, c.y)); }
__device__ __forceinline__ float tneg(float a) { return -a; }
__device__ __forceinline__ float2 tneg(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ double tneg(double a) { return -a; }
__device__ __forceinline__ double2 tneg(double2 a) { return make_double2(-a.x, -a.y); }
// |a| > thr (a part's magnitude, thr >= 0 as bits) without the FP64 pipe
__device__ __forceinline__ bool above(double a, long long thr) { return (__double_as_longlong(a) & 0x7fffffffffffffffll) > thr; }
__device__ __forceinline__ bool above(double2 a, long long thr) { return above(a.x, thr) || above(a.y, thr); }

template <typename T>
__device__ bool jacobi(T* A, T* V, int M, float tol, int max_sweeps) {
  using RT = decltype(tre(T{}));
  constexpr bool F64 = sizeof(RT) == 8;
  constexpr int kABlocks = (kMaxGramDim / 2) * (kMaxGramDim / 2 + 1);   // half blocks of A at most
  constexpr int kAThreads = 96;
  constexpr int kAItems = (kABlocks + kAThreads - 1) / kAThreads;
  constexpr int kVThreads = kEigThreads - kAThreads;
  constexpr int kVItems = (kMaxGramDim / 2 * kMaxGramDim + kVThreads - 1) / kVThreads;
  __shared__ Rot<T> rot[kMaxGramDim / 2];
  __shared__ int more;
  const int tid = threadIdx.x, lane = tid & 31;
  const int Mp = M + (M & 1), nb = Mp / 2;
  const int na = nb * (nb + 1), nv = nb * M;
  const bool fora = tid < kAThreads;
  // this thread's items: (i, j, column of pair j) of A, or (pair j, row k) of V
  constexpr int kItems = kAItems > kVItems ? kAItems : kVItems;
  int it_i[kItems], it_j[kItems];
#pragma unroll
  for (int q = 0; q < kItems; ++q) {
    it_i[q] = it_j[q] = -1;
    if (fora) {
      const int w = tid + q * kAThreads;
      if (q < kAItems && w < na) { tri_pq(w >> 1, nb, &it_i[q], &it_j[q]); it_j[q] = 2 * it_j[q] + (w & 1); }
    } else {
      const int w = tid - kAThreads + q * kVThreads;
      if (q < kVItems && w < nv) { it_j[q] = w / M; it_i[q] = w % M; }
    }
  }
  auto pair_of = [&](int st, int i, int* p, int* q) {
    int a = st, c = Mp - 1;
    if (i > 0) {
      a = st + i;
      if (a >= Mp - 1) a -= Mp - 1;
      c = st - i;
      if (c < 0) c += Mp - 1;
    }
    *p = a < c ? a : c;
    *q = a < c ? c : a;
  };
  for (int sweep = 0; sweep < max_sweeps; ++sweep) {
    float dmax = lane < M ? fabsf((float)tre(A[lane * kJP + lane])) : 0.f;
#pragma unroll
    for (int o = 16; o; o >>= 1) dmax = fmaxf(dmax, __shfl_xor_sync(0xffffffffu, dmax, o));
    const float floor2 = kFloor32 * dmax * kFloor32 * dmax;
    const long long thr = __double_as_longlong((double)(tol * dmax));
    bool did = false, big = false;
    for (int st = 0; st < Mp - 1; ++st) {
      bool rotates = false;
      T apq = tscal<T>(0.0);
      RT app = RT(0), aqq = RT(0);
      if (lane < nb) {
        int p, q;
        pair_of(st, lane, &p, &q);
        if (q < M) {
          apq = A[p * kJP + q];
          if constexpr (F64) {
            rotates = above(apq, thr);
            if (rotates && tid < 32) { app = tre(A[p * kJP + p]); aqq = tre(A[q * kJP + q]); }
          } else {
            app = tre(A[p * kJP + p]);
            aqq = tre(A[q * kJP + q]);
            const float a2 = tabs2(apq);
            rotates = a2 > tol * tol * fabsf(app * aqq) && a2 > floor2;
          }
        }
      }
      const unsigned any = __ballot_sync(0xffffffffu, rotates);
      if (!any) continue;                                // the same on every warp
      did = true;
      if (tid < 32 && rotates) {
        const float a2 = tabs2(to32f(apq));
        const float inv = rsqrtf(a2);
        const float th = 0.5f * (float)(aqq - app) * inv;
        const float h2 = 1.f + th * th;
        const float tf = copysignf(__fdividef(1.f, fabsf(th) + h2 * rsqrtf(h2)), th);
        big |= fabsf(tf) > 2e-4f;
        Rot<T> r;
        T ph;
        if constexpr (F64) {
          const double t = tf, h = fma(t, t, 1.0), hh = -0.5 * h;
          double y = rsqrtf(fmaf(tf, tf, 1.f));          // 1 / sqrt(h): two Newton steps in FP64
          y = y * fma(hh * y, y, 1.5);
          y = y * fma(hh * y, y, 1.5);
          r.c = y;
          r.s = t * y;
          ph = unit_phase(apq);
        } else {
          r.c = rsqrtf(1.f + tf * tf);
          r.s = tf * r.c;
          ph = tscale(tconj(apq), inv);
        }
        r.sp = tscale(ph, r.s);
        r.cp = tscale(ph, r.c);
        rot[lane] = r;
      }
      __syncthreads();                                   // rotations written, pairs read by every warp
      if (fora) {
#pragma unroll
        for (int q0 = 0; q0 < kAItems; ++q0) {
          // a block's two columns are two neighbouring lanes: both read the whole
          // block before either writes
          if (q0 * kAThreads >= na) break;               // the same on every thread
          const int i = max(it_i[q0], 0), j = max(it_j[q0], 0) >> 1, col = it_j[q0] & 1;
          const bool ri = (any >> i) & 1, rj = (any >> j) & 1;
          int p, q, u, v;
          pair_of(st, i, &p, &q);
          pair_of(st, j, &u, &v);
          const bool qi = q < M, vj = v < M;
          const bool on = it_i[q0] >= 0 && (ri || rj) && (vj || !col);
          const T z = tscal<T>(0.0);
          T x0 = z, x1 = z, w0 = z, w1 = z;
          if (on) {
            x0 = A[p * kJP + u];
            if (qi) x1 = A[q * kJP + u];
            if (vj) w0 = A[p * kJP + v];
            if (qi && vj) w1 = A[q * kJP + v];
          }
          __syncwarp();
          if (!on) continue;
          // column `col` of X R, then R^H of it
          if (rj) {
            const Rot<T> r = rot[j];
            const RT f = col ? r.s : r.c;
            const T g = col ? r.cp : tneg(r.sp);
            x0 = cmacc(g, w0, tscale(x0, f));
            x1 = cmacc(g, w1, tscale(x1, f));
          } else if (col) {
            x0 = w0;
            x1 = w1;
          }
          if (ri) {
            const Rot<T> r = rot[i];
            const T y0 = x0, y1 = x1;
            x0 = cmacc(tneg(tconj(r.sp)), y1, tscale(y0, r.c));
            x1 = cmacc(tconj(r.cp), y1, tscale(y0, r.s));
          }
          const int uc = col ? v : u;
          if (i != j) {
            A[p * kJP + uc] = x0;
            A[uc * kJP + p] = tconj(x0);
            if (qi) { A[q * kJP + uc] = x1; A[uc * kJP + q] = tconj(x1); }
          } else if (col == 0) {
            A[p * kJP + p] = tscal<T>(tre(x0));
          } else {
            if (!F64) x0 = z;                            // the rotated pair: zero by construction
            A[p * kJP + q] = x0;
            A[q * kJP + p] = tconj(x0);
            A[q * kJP + q] = tscal<T>(tre(x1));
          }
        }
      } else {
#pragma unroll
        for (int q0 = 0; q0 < kVItems; ++q0) {
          const int j = it_j[q0], k = it_i[q0];
          if (j < 0) break;
          if (!((any >> j) & 1)) continue;
          int u, v;
          pair_of(st, j, &u, &v);
          const Rot<T> r = rot[j];
          const T x = V[k * kJP + u], y = V[k * kJP + v];
          V[k * kJP + u] = cmacc(tneg(r.sp), y, tscale(x, r.c));
          V[k * kJP + v] = cmacc(r.cp, y, tscale(x, r.s));
        }
      }
      __syncthreads();
    }
    if (!did) return true;                               // no rotation in the whole sweep (the same on every thread)
    if constexpr (!F64) {
      if (tid < 32) {
        const bool b = __any_sync(0xffffffffu, big);
        if (lane == 0) more = b;
      }
      __syncthreads();
      if (!more) return true;
    }
  }
  return false;
}

constexpr float kRefined = 3e-5f;        // largest |Z| (Frobenius) refine() takes

// One refinement of an approximate eigenbasis Q (columns) of G: the W = I + Z
// with W^H (Q^H Q) W = I and W^H (Q^H G Q) W diagonal, Q <- Q W.  With R = Q^H
// Q - I and B = Q^H G Q = D + E (D its diagonal), the first-order solution is
// Z_ij = (E_ij - D_j R_ij) / (D_j - D_i), Z_ii = -R_ii / 2 (as in Ogita and
// Aishima's refinement, Japan J. Indust. Appl. Math. 35, 2018); it takes the only
// FP64 products (Q^H Q, G Q, Q^H G Q, Q Z).  What it leaves is of second order
// and up, small enough to be formed in FP32: delta solves the same linear system
// against the nonlinear terms F1 = Z^H Z + R Z + Z^H R + Z^H R Z and F2 = Z^H E +
// E Z + Z^H B Z, by fixed-point iteration with Z <- Z + delta.  Pairs of one tie
// cluster (within kTieTol of each other and coupled by less than a tenth of it)
// are not separated -- the cluster's basis is chosen afterwards from its
// projector -- only made orthonormal.  Declines (returns false, P then holds Q^H
// Q - I) when the correction is not small, |Z| >= kRefined, or the
// couplings left in tie clusters are not small against the other gaps: delta
// converges by those two ratios.
// Q's entries are multiples of 2^-26 (quantum), so R is exact, and the refined
// basis is left as Q and the correction Q Z in Y, 2^-53 of which is at most 2^-68:
// a rounding of it in FP64 would be the same for every row of L.
// Buffers: P, Z FP64; f32 five M x kJP FP32 matrices.  lam: the eigenvalues.
template <typename T, typename T32>
__device__ bool refine(const double2* G, const T* Q, T* Y, T* P, T* Z, T32* f32, int M, double* lam) {
  __shared__ double dD[kMaxGramDim], dR[kMaxGramDim];
  __shared__ float fD[kMaxGramDim];
  __shared__ float red[3][kEigThreads / 32];
  const int tid = threadIdx.x, MM = M * M, pairs = M * (M - 1) / 2;
  T32 *z32 = f32, *e32 = f32 + kMaxGramDim * kJP, *r32 = e32 + kMaxGramDim * kJP, *u32 = r32 + kMaxGramDim * kJP,
      *v32 = u32 + kMaxGramDim * kJP;
  for (int i = tid; i < MM; i += kEigThreads) {           // Y = G Q
    const int r = i / M, c = i % M;
    T acc = tscal<T>(0.0);
    for (int k = 0; k < M; ++k) acc = cmacc(gsm<T>(G[r * kJP + k]), Q[k * kJP + c], acc);
    Y[r * kJP + c] = acc;
  }
  __syncthreads();
  for (int i = tid; i < pairs + M; i += kEigThreads) {    // B above the diagonal of P, R below, both diagonals
    int r, c;
    tri_pq(i, M, &r, &c);
    T bb = tscal<T>(0.0), rr = tscal<T>(r == c ? -1.0 : 0.0);
    for (int k = 0; k < M; ++k) {
      const T q = tconj(Q[k * kJP + r]);
      bb = cmacc(q, Y[k * kJP + c], bb);
      rr = cmacc(q, Q[k * kJP + c], rr);
    }
    if (r == c) {
      dD[r] = tre(bb);
      fD[r] = (float)tre(bb);
      dR[r] = tre(rr);
      e32[r * kJP + r] = tscal<T32>(0.0);
      r32[r * kJP + r] = tscal<T32>(tre(rr));
    } else {
      P[r * kJP + c] = bb;
      P[c * kJP + r] = rr;
      e32[r * kJP + c] = to32f(bb);
      e32[c * kJP + r] = tconj(to32f(bb));
      r32[r * kJP + c] = to32f(rr);
      r32[c * kJP + r] = tconj(to32f(rr));
    }
  }
  __syncthreads();
  float dmax = (tid & 31) < M ? fabsf((float)dD[tid & 31]) : 0.f;
#pragma unroll
  for (int o = 16; o; o >>= 1) dmax = fmaxf(dmax, __shfl_xor_sync(0xffffffffu, dmax, o));
  const float tie = (float)kTieTol * dmax;
  auto tied = [&](float gap, int i, int j) { return fabsf(gap) <= tie && tabs2(e32[i * kJP + j]) <= 0.01f * tie * tie; };
  float zs = 0.f, et = 0.f, gap = 3e38f;                  // |Z|^2, largest tied coupling, smallest other gap
  for (int i = tid; i < pairs + M; i += kEigThreads) {
    int r, c;
    tri_pq(i, M, &r, &c);
    if (r == c) {
      Z[r * kJP + r] = tscal<T>(-0.5 * dR[r]);
      z32[r * kJP + r] = tscal<T32>(-0.5 * dR[r]);
      continue;
    }
    const T E = P[r * kJP + c], Rr = P[c * kJP + r];
    T zrc, zcr;
    const double dg = dD[c] - dD[r];
    const float gf = (float)dg, gi = __frcp_rn(gf);
    if (tied(gf, r, c)) {
      zrc = tscale(Rr, -0.5);
      zcr = tconj(zrc);
      et = fmaxf(et, tabs2(to32f(E)));
    } else {
      gap = fminf(gap, fabsf(gf));
      // (E - D_c R) / gap: an FP32 quotient and one correction from its FP64 remainder
      const T num = rmacc(-dD[c], Rr, E);
      zrc = to64(tscale(to32f(num), gi));
      zrc = tadd(zrc, to64(tscale(to32f(rmacc(-dg, zrc, num)), gi)));
      zcr = tconj(tadd(tscale(Rr, -1.0), tscale(zrc, -1.0)));   // Z + Z^H = -R
    }
    Z[r * kJP + c] = zrc;
    Z[c * kJP + r] = zcr;
    const T32 f = to32f(zrc);
    z32[r * kJP + c] = f;
    z32[c * kJP + r] = to32f(zcr);
    zs += 2.f * tabs2(f);
  }
#pragma unroll
  for (int o = 16; o; o >>= 1) {
    zs += __shfl_xor_sync(0xffffffffu, zs, o);
    et = fmaxf(et, __shfl_xor_sync(0xffffffffu, et, o));
    gap = fminf(gap, __shfl_xor_sync(0xffffffffu, gap, o));
  }
  if ((tid & 31) == 0) { red[0][tid >> 5] = zs; red[1][tid >> 5] = et; red[2][tid >> 5] = gap; }
  __syncthreads();
  zs = 0.f;
#pragma unroll
  for (int w = 0; w < kEigThreads / 32; ++w) {
    zs += red[0][w];
    et = fmaxf(et, red[1][w]);
    gap = fminf(gap, red[2][w]);
  }
  if (!(zs < kRefined * kRefined) || !(sqrtf(et) * 1000.f <= gap)) {   // the same on every thread
    for (int i = tid; i < pairs + M; i += kEigThreads) {  // R in both halves of P
      int r, c;
      tri_pq(i, M, &r, &c);
      if (r == c) P[r * kJP + r] = tscal<T>(dR[r]);
      else { const T v = P[c * kJP + r]; P[r * kJP + c] = v; P[c * kJP + r] = tconj(v); }
    }
    __syncthreads();
    return false;
  }
  // delta: each pass gains a factor |Z|; passes until what is left is below 1e-17
  const int passes = zs < 4e-12f ? 1 : 2;
  for (int it = 0; it < passes; ++it) {
    // u = R Z, v = E Z (not B Z: taking D Z off it again leaves an FP32 rounding of D Z,
    // of first order, in terms of second; divided by the gap at the cut it put the trace
    // of nine iterations of Grover's search at rank 4, 8 and 9 qubits, 1.6e-13 off, rms
    // against long double, now 1.9e-14, as through L')
    for (int i = tid; i < 2 * MM; i += kEigThreads) {
      const int which = i >= MM, k = which ? i - MM : i, r = k / M, c = k % M;
      const T32* X = which ? e32 : r32;
      T32 acc = tscal<T32>(0.0);
      for (int q = 0; q < M; ++q) acc = cmacc(X[r * kJP + q], z32[q * kJP + c], acc);
      (which ? v32 : u32)[r * kJP + c] = acc;
    }
    __syncthreads();
    T32 zn[(kMaxGramDim * (kMaxGramDim + 1) / 2 + kEigThreads - 1) / kEigThreads][2];
    int slot = 0;
#pragma unroll
    for (int i0 = 0; i0 < kMaxGramDim * (kMaxGramDim + 1) / 2; i0 += kEigThreads, ++slot) {
      const int i = i0 + tid;
      if (i >= pairs + M) continue;
      int r, c;
      tri_pq(i, M, &r, &c);
      T32 f1 = tadd(u32[r * kJP + c], tconj(u32[c * kJP + r]));
      T32 f2 = tadd(v32[r * kJP + c], tconj(v32[c * kJP + r]));
      for (int k = 0; k < M; ++k) {
        const T32 zk = tconj(z32[k * kJP + r]), zc = z32[k * kJP + c];
        f1 = cmacc(zk, tadd(zc, u32[k * kJP + c]), f1);
        f2 = cmacc(zk, rmacc(fD[k], zc, v32[k * kJP + c]), f2);
      }
      if (r == c) {
        const float dl = -0.5f * tre(f1);
        zn[slot][0] = tscal<T32>(dl);
        lam[r] = dD[r] + 2.0 * (double)tre(Z[r * kJP + r]) * dD[r] + (double)tre(f2) + 2.0 * (double)dl * dD[r];
      } else {
        T32 d;
        const float gf = (float)(dD[c] - dD[r]);
        if (tied(gf, r, c)) d = tscale(f1, -0.5f);
        else d = tscale(tadd(f2, tscale(f1, -(float)dD[c])), __frcp_rn(gf));
        zn[slot][0] = d;
        zn[slot][1] = tconj(tadd(tscale(f1, -1.f), tscale(d, -1.f)));
      }
    }
    __syncthreads();
    // Z = first order + delta; the FP32 copy for the next pass
    slot = 0;
#pragma unroll
    for (int i0 = 0; i0 < kMaxGramDim * (kMaxGramDim + 1) / 2; i0 += kEigThreads, ++slot) {
      const int i = i0 + tid;
      if (i >= pairs + M) continue;
      int r, c;
      tri_pq(i, M, &r, &c);
      const bool end = it + 1 == passes;
      const T zr = tadd(Z[r * kJP + c], to64(zn[slot][0]));
      if (end) Z[r * kJP + c] = zr;
      else z32[r * kJP + c] = to32f(zr);
      if (r != c) {
        const T zc = tadd(Z[c * kJP + r], to64(zn[slot][1]));
        if (end) Z[c * kJP + r] = zc;
        else z32[c * kJP + r] = to32f(zc);
      }
    }
    __syncthreads();
  }
  for (int i = tid; i < MM; i += kEigThreads) {           // Y = Q Z
    const int r = i / M, c = i % M;
    T acc = tscal<T>(0.0);
    for (int k = 0; k < M; ++k) acc = cmacc(Q[r * kJP + k], Z[k * kJP + c], acc);
    Y[r * kJP + c] = acc;
  }
  __syncthreads();
  return true;
}

// The nearest multiple of 2^-26 (|x| < 2^25): products of two such numbers of at
// most 1 are multiples of 2^-52, and so are their sums: exact in FP64.
__device__ __forceinline__ double quantum(double x) { return __dadd_rn(__dadd_rn(x, 0x1.8p26), -0x1.8p26); }
__device__ __forceinline__ double2 quantum(double2 x) { return make_double2(quantum(x.x), quantum(x.y)); }

// An eigenbasis in columns (pitch kJP): hi, or hi + lo with hi in multiples of 2^-26
// (lo null: hi alone); sum: rounded to FP64.  unit: the columns' norms are off by
// the roundings of the FP64 Jacobi.
template <typename T> struct Basis { T *hi, *lo, *sum; bool unit; };

// (hi + lo) u for the phase u, unit to FP64's rounding: u too is split at 2^-26, its
// norm's error, found exactly, goes into the low part.
__device__ __forceinline__ void turn(double hi, double lo, double u, double* bh, double* bl) { *bh = hi * u; *bl = lo * u; }
__device__ __forceinline__ void turn(double2 hi, double2 lo, double2 u, double2* bh, double2* bl) {
  const double2 uq = quantum(u), ul = make_double2(u.x - uq.x, u.y - uq.y);
  const double off = fma(uq.x, uq.x, fma(uq.y, uq.y, -1.0)) + fma(2.0 * uq.x + ul.x, ul.x, (2.0 * uq.y + ul.y) * ul.y);
  *bh = cmacc(hi, uq, make_double2(0.0, 0.0));
  *bl = cmacc(hi, ul, cmacc(lo, u, make_double2(-0.5 * off * bh->x, -0.5 * off * bh->y)));
}
// After the eigensolver: eigenvalues lam sorted descending (ties keep index
// order), clusters of ties given a canonical basis, and the outputs W = first
// keep canonical eigenvectors (basis + low, columns, pitch kJP; rounded, M x keep
// complex, in W), lam_out (sorted), keep and the scale.  T is double (real G: real
// eigenvectors, real arithmetic) or double2.  Candidate j of a cluster with
// eigenvectors S is P e_j, P = S S^dagger, minus its components along the
// cluster's accepted vectors q_t; as the q_t lie in range(P),
// <q_t, P e_j> = conj(q_t[j]) and |P e_j - ...|^2 = P_jj - sum_t |q_t[j]|^2,
// so the projections need no dot products.  An accepted vector is
// normalised by its computed norm.  A cluster fills its own columns of the
// basis (from the index of its first eigenvalue on), so the clusters are shared
// out over the warps (lane = row).
template <typename T>
__device__ void eig_finish(const Basis<T> Q, T* basis, T* low, const double* lam_in, int M, int r, int normalize, double unscale,
                           double* __restrict__ W, double* __restrict__ lam_out, int* keep_out, double* scale_out,
                           int* status) {
  __shared__ int order[kMaxGramDim + 1], start[kMaxGramDim + 1], nclusters;
  __shared__ double lam[kMaxGramDim];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, warps = kEigThreads / 32;
  const T* V = Q.sum;
  // descending, ties in index order: position of i = how many come before it
  for (int i = tid; i < M; i += blockDim.x) {
    int pos = 0;
    for (int j = 0; j < M; ++j) pos += lam_in[j] > lam_in[i] || (lam_in[j] == lam_in[i] && j < i);
    order[pos] = i;
    lam[pos] = lam_in[i];
  }
  const int keep = r < M ? r : M;
  for (int i = tid; i < M * kJP; i += blockDim.x) basis[i] = low[i] = tscal<T>(0.0);
  __syncthreads();
  const double lam1 = lam[0] > 0.0 ? lam[0] : 0.0;
  if (tid == 0) {
    int nc = 0, i0 = 0;
    while (i0 < keep) {
      start[nc++] = i0;
      int i1 = i0 + 1;
      while (i1 < M && lam[i0] - lam[i1] <= kTieTol * lam1) ++i1;
      i0 = i1;
    }
    start[nc] = i0;
    nclusters = nc;
  }
  __syncthreads();
  for (int cl = warp; cl < nclusters; cl += warps) {
    const int i0 = start[cl], i1 = start[cl + 1];
    const int s = i1 - i0;
    int found = i0;
    if (s == 1) {
      // one eigenvector v: the first candidate is P e_j = v conj(v_j) for the
      // first j with |v_j| > kGsAccept, normalised: v times a phase
      const int col = order[i0];
      const T vl = lane < M ? V[lane * kJP + col] : tscal<T>(0.0);
      const unsigned ok = __ballot_sync(0xffffffffu, lane < M && tabs2(vl) > kGsAccept * kGsAccept);
      if (ok) {
        const T ph = unit_phase(V[(__ffs(ok) - 1) * kJP + col]);
        T b = tscal<T>(0.0), bl = b;
        if (lane < M) {
          if (Q.lo) turn(Q.hi[lane * kJP + col], Q.lo[lane * kJP + col], ph, &b, &bl);
          else b = tmul(vl, ph);
        }
        if (Q.unit) {                                      // the norm's error into the low part
          double n2 = lane < M ? tabs2(b) : 0.0;
          if (lane == 0) n2 -= 1.0;
#pragma unroll
          for (int o = 16; o; o >>= 1) n2 += __shfl_xor_sync(0xffffffffu, n2, o);
          bl = tscale(b, -0.5 * n2);
        }
        if (lane < M) {
          basis[lane * kJP + i0] = b;
          low[lane * kJP + i0] = bl;
        }
        continue;
      }
    }
    // P = S S^dagger; GS of P e_j, j = 0..M-1, thresholds kGsAccept then
    // kGsFallback, as far as the kept vectors go
    const int need = i1 < keep ? i1 : keep;
    for (int pass = 0; pass < 2 && found < need; ++pass) {
      const double thr = pass == 0 ? kGsAccept : kGsFallback;
      for (int j = 0; j < M && found < need; ++j) {
        // row `lane` of P e_j and of the accepted vectors' parts, and this lane's
        // share of P_jj - sum_t |q_t[j]|^2 (lane = member of the cluster)
        double n2 = lane < s ? tabs2(V[j * kJP + order[i0 + lane]]) : 0.0;
        if (lane < found - i0) n2 -= tabs2(basis[j * kJP + i0 + lane]);
        T v0 = tscal<T>(0.0), v1 = tscal<T>(0.0);
        if (lane < M) {
          for (int c = 0; c < s; c += 2) {
            const int ca = order[i0 + c];
            v0 = cmacc(V[lane * kJP + ca], tconj(V[j * kJP + ca]), v0);
            if (c + 1 < s) {
              const int cb = order[i0 + c + 1];
              v1 = cmacc(V[lane * kJP + cb], tconj(V[j * kJP + cb]), v1);
            }
          }
          for (int t = i0; t < found; t += 2) {
            v0 = cmacc(basis[lane * kJP + t], tneg(tconj(basis[j * kJP + t])), v0);
            if (t + 1 < found) v1 = cmacc(basis[lane * kJP + t + 1], tneg(tconj(basis[j * kJP + t + 1])), v1);
          }
        }
        const T v = tadd(v0, v1);
        double nv = lane < M ? tabs2(v) : 0.0;
#pragma unroll
        for (int o = 16; o; o >>= 1) {
          n2 += __shfl_xor_sync(0xffffffffu, n2, o);
          nv += __shfl_xor_sync(0xffffffffu, nv, o);
        }
        if (n2 > thr * thr) {
          if (lane < M) basis[lane * kJP + found] = tscale(v, rsqrt(nv));
          ++found;
          __syncwarp();
        }
      }
    }
    if (found < need && lane == 0) status[0] = 2;      // incomplete cluster
  }
  __syncthreads();
  // outputs
  for (int i = tid; i < M * keep; i += blockDim.x) {
    const int p = i / keep, c = i % keep;
    const T v = tadd(basis[p * kJP + c], low[p * kJP + c]);
    if constexpr (sizeof(T) == 16) {
      W[2 * (p * keep + c)] = v.x;
      W[2 * (p * keep + c) + 1] = v.y;
    } else {
      W[2 * (p * keep + c)] = v;
      W[2 * (p * keep + c) + 1] = 0.0;
    }
  }
  for (int i = tid; i < M; i += blockDim.x) lam_out[i] = lam[i] * unscale;
  if (tid == 0) {
    double kept = 0.0;
    for (int i = 0; i < keep; ++i) kept += lam[i] * unscale;
    keep_out[0] = keep;
    scale_out[0] = normalize ? 1.0 / sqrt(kept) : 1.0;
  }
}

// Shared memory of the eigensolver: G, four FP64 matrices, five FP32 ones
constexpr size_t kEigMat = (size_t)kMaxGramDim * kJP;
constexpr int kEigSmem = (int)(kEigMat * (5 * sizeof(double2) + 5 * sizeof(float2)));
constexpr float kTol32 = 3e-7f;

// Eigenvalues lam and eigenvectors of G; see eig_member.  Q, Y, P, Z: matrices; G's
// space may hold the basis afterwards.
template <typename T, typename T32>
__device__ Basis<T> eig_vectors(double2* G, T* Q, T* Y, T* P, T* Z, T32* f32, int M, double* lam, int* status) {
  T32 *A32 = f32, *V32 = f32 + kEigMat;
  const int tid = threadIdx.x, MM = M * M;
  for (int i = tid; i < MM; i += kEigThreads) {
    const int p = i / M, q = i % M;
    A32[p * kJP + q] = to32(gsm<T>(G[p * kJP + q]));
    V32[p * kJP + q] = tscal<T32>(p == q ? 1.0 : 0.0);
  }
  __syncthreads();
  jacobi<T32>(A32, V32, M, kTol32, kJacobiSweeps32);    // not converging here only costs FP64 sweeps
  for (int i = tid; i < MM; i += kEigThreads) Q[(i / M) * kJP + i % M] = quantum(to64(V32[(i / M) * kJP + i % M]));
  __syncthreads();
  if (refine<T, T32>(G, Q, Y, P, Z, f32, M, lam)) {
    T* S = reinterpret_cast<T*>(G);
    for (int i = tid; i < MM; i += kEigThreads) {
      const int at = (i / M) * kJP + i % M;
      S[at] = tadd(Q[at], Y[at]);
    }
    return Basis<T>{Q, Y, S, false};
  }
  {
    for (int i = tid; i < MM; i += kEigThreads) {          // Z = -R / 2 + 3 R^2 / 8 (R^2 in FP32: it is 1e-12)
      const int rr = i / M, c = i % M;
      T32 acc = tscal<T32>(0.0);
      for (int k = 0; k < M; ++k) acc = cmacc(to32f(P[rr * kJP + k]), to32f(P[k * kJP + c]), acc);
      Z[rr * kJP + c] = tadd(tscale(P[rr * kJP + c], -0.5), to64(tscale(acc, 0.375f)));
    }
    __syncthreads();
    for (int i = tid; i < MM; i += kEigThreads) {          // Y = Q + Q Z
      const int rr = i / M, c = i % M;
      T acc = Q[rr * kJP + c];
      for (int k = 0; k < M; ++k) acc = cmacc(Q[rr * kJP + k], Z[k * kJP + c], acc);
      Y[rr * kJP + c] = acc;
    }
    __syncthreads();
    T* t = Q;
    Q = Y;
    Y = t;
    for (int i = tid; i < MM; i += kEigThreads) {          // P = G Q
      const int rr = i / M, c = i % M;
      T acc = tscal<T>(0.0);
      for (int k = 0; k < M; ++k) acc = cmacc(gsm<T>(G[rr * kJP + k]), Q[k * kJP + c], acc);
      P[rr * kJP + c] = acc;
    }
    __syncthreads();
    for (int i = tid; i < MM; i += kEigThreads) {          // Y = Q^dagger P, upper triangle, mirrored
      const int rr = i / M, c = i % M;
      if (rr > c) continue;
      T acc = tscal<T>(0.0);
      for (int k = 0; k < M; ++k) acc = cmacc(tconj(Q[k * kJP + rr]), P[k * kJP + c], acc);
      if (rr == c) acc = tscal<T>(tre(acc));
      Y[rr * kJP + c] = acc;
      Y[c * kJP + rr] = tconj(acc);
    }
    __syncthreads();
    if (!jacobi<T>(Y, Q, M, (float)kRotTol, kJacobiSweeps) && tid == 0) status[0] = 1;
    __syncthreads();
    for (int i = tid; i < M; i += kEigThreads) lam[i] = tre(Y[i * kJP + i]);
  }
  return Basis<T>{Q, nullptr, Q, true};
}

// Eigendecomposition of G (Hermitian, M x M, in shared memory, scaled to a
// largest diagonal entry in [1, 2)), then eig_finish.  The FP32 Jacobi gives a
// basis to about 1e-6; refine() makes it FP64-accurate with four FP64 matrix
// products.  Where it declines (close eigenvalues outside a tie cluster, as the
// symmetric noise of Grover's search makes them) the basis is made orthonormal,
// Q (I - R / 2 + 3 R^2 / 8) with R = Q^dagger Q - I (an error of |R|^3, 1e-18), and
// the FP64 Jacobi takes Q^dagger G Q, nearly diagonal by then.  The kept canonical
// eigenvectors are *basis + *low (columns, pitch kJP, shared memory).
template <typename T, typename T32>
__device__ void eig_member(T** basis, T** low, double2* G, bool diagonal, int M, int r, int normalize, double unscale, double* __restrict__ W,
                         double* __restrict__ lam_out, int* keep, double* scale, int* status) {
  __shared__ double lam[kMaxGramDim];
  T* Q = reinterpret_cast<T*>(G + kEigMat);
  T* Y = reinterpret_cast<T*>(G + 2 * kEigMat);
  T* P = reinterpret_cast<T*>(G + 3 * kEigMat);
  T* Z = reinterpret_cast<T*>(G + 4 * kEigMat);
  T32* f32 = reinterpret_cast<T32*>(G + 5 * kEigMat);
  const int tid = threadIdx.x, MM = M * M;
  Basis<T> B{Q, nullptr, Q, false};
  if (diagonal) {
    for (int i = tid; i < MM; i += kEigThreads) {
      const int p = i / M, q = i % M;
      Q[p * kJP + q] = tscal<T>(p == q ? 1.0 : 0.0);
      if (p == q) lam[p] = G[p * kJP + p].x;
    }
  } else {
    B = eig_vectors<T, T32>(G, Q, Y, P, Z, f32, M, lam, status);
  }
  __syncthreads();
  eig_finish<T>(B, P, Z, lam, M, r, normalize, unscale, W, lam_out, keep, scale, status);
  *basis = P;
  *low = Z;
}

// Where k_eig_truncate takes its Gram matrices from: the members' blocks
// (k_gram_reduce; form 0), or the moments of a dense one-qubit (1) or a diagonal
// (2) channel with its Kraus operators (E + b e_stride).
struct EigSource {
  int form;
  int kq, K;                             // target qubits, Kraus operators
  int blocks, groups;                    // the member's rows of partial sums: per row block, then per group
  int estride;
  const double* partials;
  const double* E;
  int e_stride;
  int real;                              // the moments are real
};

extern __shared__ double2 eig_sm[];

// One block per member: G_b, its eigendecomposition (real arithmetic when G_b
// is real), truncation to r_b (or to trunc_r > 0 for an explicit truncation),
// keep_b recorded; with moments, also the matrices V_ij of the projection.
// One SM works while the others wait, so it is latency that counts.  A real 16 x
// 16 matrix (rank 8, two Kraus operators) took 126 us with 256 threads, an FP64
// Jacobi after the FP32 one and three block barriers a step.
__global__ void __launch_bounds__(kEigThreads) k_eig_truncate(double* __restrict__ small, int sstride, RankCounts rc,
                                                              int trunc_r, int normalize, int* status,
                                                              const __grid_constant__ EigSource src) {
  __shared__ double2 sE[8 * 16];
  __shared__ double2 sS[256];
  const int b = blockIdx.x, tid = threadIdx.x;
  const int M = rc.M[b];
  const int r = trunc_r > 0 ? trunc_r : rc.rank[b];
  double* base = small + (size_t)b * sstride;
  double2* G = eig_sm;
  const int D = 1 << src.kq, K = src.K;
  const int m = src.form ? M / K : M;
  const bool diag = src.form == 2;
  if (src.form == 0) {
    const double* Gin = base + kSmallG;
    for (int i = tid; i < M * M; i += kEigThreads) G[(i / M) * kJP + i % M] = make_double2(Gin[2 * i], Gin[2 * i + 1]);
  } else {
    // the moments (in Z's space), the Kraus operators, S^ab = E_a^dagger E_b
    double2* Tm = G + 4 * kEigMat;
    const int ne = mom_entries(m, D, diag);
    const double* part = src.partials + ((size_t)b * (src.blocks + src.groups) + src.blocks) * src.estride;
    for (int i = tid; i < ne; i += kEigThreads) {
      double re[kMomGroups], im[kMomGroups];
#pragma unroll
      for (int k = 0; k < kMomGroups; ++k) {
        const double* p = part + (size_t)k * src.estride;
        re[k] = im[k] = 0.0;
        if (k < src.groups) {
          if (src.real) re[k] = __ldcg(p + i);
          else { const double2 v = __ldcg(reinterpret_cast<const double2*>(p) + i); re[k] = v.x; im[k] = v.y; }
        }
      }
      double sr = 0.0, si = 0.0;
#pragma unroll
      for (int k = 0; k < kMomGroups; ++k) { sr += re[k]; si += im[k]; }
      Tm[i] = make_double2(sr, si);
    }
    const double* Eb = src.E + (size_t)b * src.e_stride;
    for (int i = tid; i < K * D * D; i += kEigThreads) sE[i] = make_double2(__ldcg(Eb + 2 * i), __ldcg(Eb + 2 * i + 1));
    __syncthreads();
    const int per = diag ? D : D * D;
    for (int i = tid; i < K * K * per; i += kEigThreads) {
      const int ab = i / per, ij = i % per, ka = ab / K, kb = ab % K;
      double2 acc = make_double2(0.0, 0.0);
      if (diag) {
        acc = zmul(zconj(sE[(ka * D + ij) * D + ij]), sE[(kb * D + ij) * D + ij]);
      } else {
        for (int row = 0; row < D; ++row)
          acc = cmacc(zconj(sE[(ka * D + row) * D + ij / D]), sE[(kb * D + row) * D + ij % D], acc);
      }
      sS[i] = acc;
    }
    __syncthreads();
    const int tri = m * (m + 1) / 2;
    auto moment = [&](int l, int p, int q) {
      const bool up = p <= q;
      const int x = up ? p : q, y = up ? q : p;
      const double2 v = Tm[l * tri + x * m - x * (x - 1) / 2 + (y - x)];
      return up ? v : zconj(v);
    };
    for (int i = tid; i < M * (M + 1) / 2; i += kEigThreads) {
      int row, col;
      tri_pq(i, M, &row, &col);
      const int ka = row / m, p = row % m, kb = col / m, q = col % m;
      const double2* S = sS + (ka * K + kb) * per;
      double2 g = make_double2(0.0, 0.0);
      if (diag) {
        for (int l = 0; l < D; ++l) g = cmacc(S[l], moment(l, p, q), g);
      } else {
        g = cmacc(S[0], moment(0, p, q), g);
        g = cmacc(S[3], moment(1, p, q), g);
        g = cmacc(S[1], Tm[2 * tri + p * m + q], g);
        g = cmacc(S[2], zconj(Tm[2 * tri + q * m + p]), g);
      }
      if (row == col) g.y = 0.0;
      G[row * kJP + col] = g;
      G[col * kJP + row] = zconj(g);
    }
  }
  __syncthreads();
  // scale by a power of two: the FP32 stages work on entries of order 1
  int hi = (tid & 31) < M ? __double2hiint(G[(tid & 31) * (kJP + 1)].x) : 0, cplx = 0;
#pragma unroll
  for (int o = 16; o; o >>= 1) hi = max(hi, __shfl_xor_sync(0xffffffffu, hi, o));
  const int be = hi >> 20;                               // the largest diagonal entry's biased exponent
  const bool scaled = be > 64 && be < 1984;
  const double down = scaled ? __hiloint2double((2046 - be) << 20, 0) : 1.0;
  const double unscale = scaled ? __hiloint2double(be << 20, 0) : 1.0;
  __syncthreads();
  for (int i = tid; i < M * M; i += kEigThreads) {
    double2& g = G[(i / M) * kJP + i % M];
    g = make_double2(g.x * down, g.y * down);
    cplx |= g.y != 0.0;
  }
  cplx = __syncthreads_or(cplx);
  // nothing above the FP64 Jacobi's threshold off the diagonal (every channel of a
  // rank-1 real factor): the axes are the eigenvectors
  int offdiag = 0;
  const long long thr = __double_as_longlong(kRotTol);
  for (int i = tid; i < M * M; i += kEigThreads)
    if (i / M != i % M) offdiag |= above(G[(i / M) * kJP + i % M], thr);
  const bool diagonal = !__syncthreads_or(offdiag) && scaled;
  double *W = base + kSmallW, *lam = base + kSmallLam, *scale = base + kSmallScale;
  double2 *basis_c = nullptr, *low_c = nullptr;
  double *basis_r = nullptr, *low_r = nullptr;
  if (cplx) eig_member<double2, float2>(&basis_c, &low_c, G, diagonal, M, r, normalize, unscale, W, lam, rc.keep + b, scale, status);
  else eig_member<double, float>(&basis_r, &low_r, G, diagonal, M, r, normalize, unscale, W, lam, rc.keep + b, scale, status);
  if (src.form == 0) return;
  __threadfence_block();
  __syncthreads();
  // V_ij = scale sum_a (E_a)_ij W_a, [ij][p][c], the small terms first: V's rounding
  // is the same for every row of L, and with W rounded before it the trace of a channel
  // that truncates nothing was off by 2.7e-16 (rms, random factors of 1 to 8 columns;
  // 1.7e-16 through L', now 1.1e-16, for 1.7 us more a channel)
  const int keep = r < M ? r : M;
  const double sc = normalize ? *(volatile double*)scale : 1.0;
  const int nv = diag ? D : D * D;
  double* V = base + kSmallV;
  for (int i = tid; i < nv * m * keep; i += kEigThreads) {
    const int c = i % keep, p = (i / keep) % m, ij = i / (keep * m);
    const int at = diag ? ij * D + ij : ij;
    double2 acc = make_double2(0.0, 0.0);
    for (int part = 0; part < 2; ++part) {
      const double2* wc = part ? basis_c : low_c;
      const double* wr = part ? basis_r : low_r;
      for (int a = K - 1; a >= 0; --a) {
        const int row = (a * m + p) * kJP + c;
        const double2 w = cplx ? wc[row] : make_double2(wr[row], 0.0);
        if (src.real) acc.x = fma(sE[a * D * D + at].x, w.x, acc.x);
        else acc = cmacc(sE[a * D * D + at], w, acc);
      }
    }
    if (src.real) V[i] = acc.x * sc;
    else { V[2 * i] = acc.x * sc; V[2 * i + 1] = acc.y * sc; }
  }
}

// L_b[c] = scale_b sum_p L'_b[p] W_b[p][c] for c < keep_b, columns keep_b..
// m_b - 1 cleared, then m_b = keep_b; one thread per row and member
// (grid.y), all kept columns (each element of L' is read once).  KMAX is a
// power of two >= every keep_b.  REAL: L' and W are real.
template <typename R, bool REAL, int KMAX>
__global__ void __launch_bounds__(256) k_project(const cplx<R>* __restrict__ Lp, cplx<R>* __restrict__ L, int n,
                                                 int mcap, int rcap, int K, const double* __restrict__ small,
                                                 int sstride, RankCounts rc) {
  __shared__ double2 sW[kMaxGramDim * KMAX];
  const int b = blockIdx.y;
  const int M = rc.M[b], keep = rc.keep[b];
  const int old_cols = M / K;
  const double* base = small + (size_t)b * sstride;
  const double scale = base[kSmallScale];
  const double* W = base + kSmallW;
  for (int i = threadIdx.x; i < M * KMAX; i += blockDim.x) {
    const int p = i / KMAX, c = i % KMAX;
    sW[i] = c < keep ? make_double2(W[2 * (p * keep + c)] * scale, W[2 * (p * keep + c) + 1] * scale)
                     : make_double2(0.0, 0.0);
  }
  __syncthreads();
  if (blockIdx.x == 0 && threadIdx.x == 0) rc.cols[b] = keep;
  const uint64_t N = 1ull << n;
  const cplx<R>* Lpb = Lp + (uint64_t)b * mcap * N;
  cplx<R>* Lb = L + (uint64_t)b * rcap * N;
  for (uint64_t x = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; x < N; x += (uint64_t)gridDim.x * blockDim.x) {
    if constexpr (REAL) {
      double acc[KMAX];
#pragma unroll
      for (int c = 0; c < KMAX; ++c) acc[c] = 0.0;
      for (int p = 0; p < M; ++p) {
        const double a = Lpb[(uint64_t)p * N + x].x;
#pragma unroll
        for (int c = 0; c < KMAX; ++c)
          if (c < keep) acc[c] = fma(a, sW[p * KMAX + c].x, acc[c]);   // keep: the same across the block
      }
#pragma unroll
      for (int c = 0; c < KMAX; ++c)
        if (c < keep) Lb[(uint64_t)c * N + x] = mk<R>((R)acc[c], R(0));
    } else {
      double2 acc[KMAX];
#pragma unroll
      for (int c = 0; c < KMAX; ++c) acc[c] = make_double2(0.0, 0.0);
      for (int p = 0; p < M; ++p) {
        const cplx<R> a = Lpb[(uint64_t)p * N + x];
        const double ax = a.x, ay = a.y;
#pragma unroll
        for (int c = 0; c < KMAX; ++c) {
          if (c >= keep) continue;                         // keep: the same across the block
          const double2 w = sW[p * KMAX + c];              // a * w, four FMAs
          acc[c].x = fma(ax, w.x, fma(-ay, w.y, acc[c].x));
          acc[c].y = fma(ax, w.y, fma(ay, w.x, acc[c].y));
        }
      }
#pragma unroll
      for (int c = 0; c < KMAX; ++c)
        if (c < keep) Lb[(uint64_t)c * N + x] = mk<R>((R)acc[c].x, (R)acc[c].y);
    }
    for (int c = keep; c < old_cols; ++c) Lb[(uint64_t)c * N + x] = mk<R>(R(0), R(0));
  }
}

// Blocks of a grid-stride kernel over `rows` rows per member: about four
// 256-thread blocks per SM in all, at least one per member.
unsigned rows_blocks(uint64_t rows, int members) {
  const uint64_t want = ((uint64_t)num_sms() * 4 + members - 1) / members;
  const uint64_t most = (rows + 255) / 256;
  return (unsigned)std::max<uint64_t>(1, std::min(want, most));
}

template <typename R>
cudaError_t expand_launch(qs_ctx* h, const Targets& tg, bool real, const double* E, int K,
                            int max_cols, const KrausGate& g) {
  const uint64_t work = ((1ull << h->n) >> 2) * (uint64_t)max_cols;
  const dim3 grid(rows_blocks(work, h->batch), h->batch);
  auto* l = static_cast<const cplx<R>*>(h->state);
  auto* lp = static_cast<cplx<R>*>(h->work);
  if (real) k_kraus_expand<R, true><<<grid, kExpBlock, 0, h->stream>>>(l, lp, h->n, h->rank, h->mcap, tg, E, K, h->rc, g);
  else k_kraus_expand<R, false><<<grid, kExpBlock, 0, h->stream>>>(l, lp, h->n, h->rank, h->mcap, tg, E, K, h->rc, g);
  return cudaGetLastError();
}

template <typename R, bool REAL, int KMAX>
void project_launch(qs_ctx* h, int K) {
  const dim3 grid(rows_blocks(1ull << h->n, h->batch), h->batch);
  k_project<R, REAL, KMAX><<<grid, 256, 0, h->stream>>>(static_cast<const cplx<R>*>(h->work),
                                                        static_cast<cplx<R>*>(h->state), h->n, h->mcap, h->rank, K,
                                                        h->rsmall, kRankStride, h->rc);
}

template <typename R, bool REAL>
void project_kmax(qs_ctx* h, int K, int max_keep) {
  if (max_keep <= 1) project_launch<R, REAL, 1>(h, K);
  else if (max_keep <= 2) project_launch<R, REAL, 2>(h, K);
  else if (max_keep <= 4) project_launch<R, REAL, 4>(h, K);
  else if (max_keep <= 8) project_launch<R, REAL, 8>(h, K);
  else project_launch<R, REAL, 16>(h, K);
}

}  // namespace

int gram_rows_per_block(int n) {
  const uint64_t N = 1ull << n;
  const uint64_t per = (N + (uint64_t)kGramRows * kGramTarget - 1) / ((uint64_t)kGramRows * kGramTarget);
  return (int)(per * kGramRows);
}

size_t gram_partials_doubles(int n, int members, int rank) {
  const uint64_t N = 1ull << n;
  const uint64_t blocks = (N + gram_rows_per_block(n) - 1) / gram_rows_per_block(n);
  const size_t mom = (size_t)mom_split(n, 1).blocks + kMomGroups;        // two-qubit channels have no more blocks
  return (size_t)members * std::max<size_t>(blocks * 2 * kTriMax, mom * mom_stride(rank));
}
int rank_counters() { return kMomGroups; }

cudaError_t launch_gram(qs_ctx* h, bool real, int max_M) {
  const uint64_t N = 1ull << h->n;
  const int rows = gram_rows_per_block(h->n);
  const int blocks = (int)((N + rows - 1) / rows);
  const dim3 grid(blocks, h->batch);
  const int nt = rows >= 16 * kGramRows ? kGramThreads : kGramThreads / 2;   // see k_gram_partials
  if (h->dtype == QS_C64 && real)
    k_gram_partials<float, true><<<grid, nt, 0, h->stream>>>((const float2*)h->work, h->n, h->mcap, rows, h->rc, h->partials);
  else if (h->dtype == QS_C64)
    k_gram_partials<float, false><<<grid, nt, 0, h->stream>>>((const float2*)h->work, h->n, h->mcap, rows, h->rc, h->partials);
  else if (real)
    k_gram_partials<double, true><<<grid, nt, 0, h->stream>>>((const double2*)h->work, h->n, h->mcap, rows, h->rc, h->partials);
  else
    k_gram_partials<double, false><<<grid, nt, 0, h->stream>>>((const double2*)h->work, h->n, h->mcap, rows, h->rc, h->partials);
  k_gram_reduce<<<dim3(max_M * (max_M + 1) / 2, h->batch), 256, 0, h->stream>>>(h->partials, blocks, h->rc, h->rsmall, kRankStride);
  return cudaGetLastError();
}

cudaError_t rank_kernel_attributes() {
  static std::atomic<bool> attr{false};
  if (attr.load()) return cudaSuccess;
  const cudaError_t e = cudaFuncSetAttribute(k_eig_truncate, cudaFuncAttributeMaxDynamicSharedMemorySize, kEigSmem);
  if (e == cudaSuccess) attr.store(true);
  return e;
}

cudaError_t launch_eig_truncate(qs_ctx* h, int trunc_r, int normalize) {
  const cudaError_t e = rank_kernel_attributes();
  if (e != cudaSuccess) return e;
  k_eig_truncate<<<h->batch, kEigThreads, kEigSmem, h->stream>>>(h->rsmall, kRankStride, h->rc, trunc_r, normalize,
                                                                 h->dstatus + 1, EigSource{});
  return cudaGetLastError();
}

namespace {
// moments, eigensolver and projection of a one-qubit or diagonal channel
template <typename R, bool REAL, int KQ, bool DIAG>
cudaError_t channel_launch(qs_ctx* h, const Targets& tg, const double* E, int K, const KrausGate& g,
                           int max_cols, int max_keep, int normalize) {
  constexpr int D = 1 << KQ, CB = 4;
  const MomSplit sp = mom_split(h->n, KQ);
  auto* L = static_cast<cplx<R>*>(h->state);
  k_moments<R, REAL, KQ, DIAG><<<dim3(sp.blocks, h->batch), kMomThreads, 0, h->stream>>>(
      L, h->n, h->rank, tg, K, h->rc, h->partials, mom_stride(h->rank), h->rcounters, h->rsmall, kRankStride, g);
  EigSource src{};
  src.form = DIAG ? 2 : 1;
  src.kq = KQ;
  src.K = K;
  src.blocks = sp.blocks;
  src.groups = (sp.blocks + kMomGroup - 1) / kMomGroup;
  src.estride = mom_stride(h->rank);
  src.partials = h->partials;
  src.E = g.k > 0 ? h->rsmall + kSmallE : E;             // a gate's set: written by k_moments
  src.e_stride = g.k > 0 ? kRankStride : 0;
  src.real = REAL ? 1 : 0;
  k_eig_truncate<<<h->batch, kEigThreads, kEigSmem, h->stream>>>(h->rsmall, kRankStride, h->rc, 0, normalize, h->dstatus + 1,
                                                                 src);
  const int nrun = max_keep <= CB ? 1 : (max_keep <= 2 * CB ? 2 : 4);
  const int per = (kProjThreads / nrun) >> KQ;           // groups of a block
  const uint64_t want = std::max<uint64_t>(1, ((1ull << h->n) >> KQ) / per);
  const uint64_t cap = (uint64_t)num_sms() * 64;         // beyond that the blocks stride
  const size_t sm = (size_t)(DIAG ? D : D * D) * max_cols * nrun * CB * (REAL ? sizeof(double) : sizeof(double2));
  k_project_fused<R, REAL, KQ, DIAG, CB><<<dim3((unsigned)std::min(want, cap), h->batch), kProjThreads, sm, h->stream>>>(
      L, h->n, h->rank, tg, K, nrun, h->rsmall, kRankStride, h->rc);
  return cudaGetLastError();
}

template <typename R, bool REAL>
cudaError_t channel_form(qs_ctx* h, const Targets& tg, bool diag, const double* E, int K, const KrausGate& g,
                         int max_cols, int max_keep, int normalize) {
  if (tg.k == 2) return channel_launch<R, REAL, 2, true>(h, tg, E, K, g, max_cols, max_keep, normalize);
  if (diag) return channel_launch<R, REAL, 1, true>(h, tg, E, K, g, max_cols, max_keep, normalize);
  return channel_launch<R, REAL, 1, false>(h, tg, E, K, g, max_cols, max_keep, normalize);
}
}  // namespace

bool gate_diagonal(const double* U, int k) {
  const int d = 1 << k;
  for (int r = 0; r < d; ++r)
    for (int c = 0; c < d; ++c)
      if (r != c && (U[2 * (r * d + c)] != 0.0 || U[2 * (r * d + c) + 1] != 0.0)) return false;
  return true;
}

cudaError_t launch_rank_channel(qs_ctx* h, const Targets& tg, bool real, bool diag, const double* E, int K,
                                const KrausGate& g, int max_cols, int max_keep, int normalize) {
  if (tg.k == 2 && !diag) {                              // through L'
    const int max_M = std::min(kMaxGramDim, K * max_cols);
    cudaError_t e = h->dtype == QS_C64 ? expand_launch<float>(h, tg, real, E, K, max_cols, g)
                                       : expand_launch<double>(h, tg, real, E, K, max_cols, g);
    if (e == cudaSuccess) e = launch_gram(h, real, max_M);
    if (e == cudaSuccess) e = launch_eig_truncate(h, 0, normalize);
    if (e == cudaSuccess) e = launch_project(h, real, K, max_keep);
    return e;
  }
  const cudaError_t e = rank_kernel_attributes();
  if (e != cudaSuccess) return e;
  if (h->dtype == QS_C64 && real) return channel_form<float, true>(h, tg, diag, E, K, g, max_cols, max_keep, normalize);
  if (h->dtype == QS_C64) return channel_form<float, false>(h, tg, diag, E, K, g, max_cols, max_keep, normalize);
  if (real) return channel_form<double, true>(h, tg, diag, E, K, g, max_cols, max_keep, normalize);
  return channel_form<double, false>(h, tg, diag, E, K, g, max_cols, max_keep, normalize);
}

cudaError_t launch_project(qs_ctx* h, bool real, int K, int max_keep) {
  if (h->dtype == QS_C64 && real) project_kmax<float, true>(h, K, max_keep);
  else if (h->dtype == QS_C64) project_kmax<float, false>(h, K, max_keep);
  else if (real) project_kmax<double, true>(h, K, max_keep);
  else project_kmax<double, false>(h, K, max_keep);
  return cudaGetLastError();
}

}  // namespace qs
