// Fidelity and trace reductions (Figs. 1-4, Eq. 10).
//
// Each member's sum is split into fixed chunks; a block reduces one chunk
// and writes an FP64 partial; a second kernel adds the partials of a member
// in a fixed order, so results are deterministic run to run.  Inside a
// thread, a complex64 state accumulates its (short) run of products in FP32
// -- each product of two FP32 numbers is formed in FP32 as the amplitudes
// are -- and everything from the warp level up is FP64.
#include <cuda_runtime.h>

#include <algorithm>

#include "internal.cuh"
#include "sums.cuh"

namespace qs {

namespace {

constexpr int kRBlock = 256;
constexpr int kChunk = 4096;            // amplitudes per block

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Block sum of (a, b); result valid in thread 0.
__device__ __forceinline__ double2 block_sum2(double a, double b) {
  __shared__ double sa[32], sb[32];
  a = warp_sum(a);
  b = warp_sum(b);
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  if (l == 0) { sa[w] = a; sb[w] = b; }
  __syncthreads();
  double2 r = make_double2(0.0, 0.0);
  if (w == 0) {
    const int nw = blockDim.x >> 5;
    a = l < nw ? sa[l] : 0.0;
    b = l < nw ? sb[l] : 0.0;
    r.x = warp_sum(a);
    r.y = warp_sum(b);
  }
  __syncthreads();
  return r;
}

// A thread's kPer amplitudes of a full chunk are read as 16-byte vectors
// (two complex64 amplitudes or one complex128) before any of them is used:
// the sweep is bound by HBM latency otherwise (one 8-byte load in flight per
// thread and iteration read 1 GiB of members at 3.3 TB/s).
constexpr int kPer = kChunk / kRBlock;   // 16 amplitudes per thread
template <typename R> struct Vec;
template <> struct Vec<float> { using T = float4; static constexpr int N = 2; };
template <> struct Vec<double> { using T = double2; static constexpr int N = 1; };
__device__ __forceinline__ float2 vget(const float4& v, int k) { return k ? make_float2(v.z, v.w) : make_float2(v.x, v.y); }
__device__ __forceinline__ double2 vget(const double2& v, int) { return v; }

// f(amplitude, reference) over the chunk starting at beg (p, r: the member's
// and the reference's first amplitude; r may be null for REF = false)
template <typename R, bool REF, typename F>
__device__ __forceinline__ void chunk_each(const cplx<R>* __restrict__ p, const cplx<R>* __restrict__ r, uint64_t beg,
                                           uint64_t N, F&& f) {
  using V = typename Vec<R>::T;
  constexpr int W = Vec<R>::N, L = kPer / W;
  if (beg + kChunk <= N) {
    const V* pv = reinterpret_cast<const V*>(p + beg) + threadIdx.x;
    const V* rv = reinterpret_cast<const V*>(r + beg) + threadIdx.x;
    V a[L];
#pragma unroll
    for (int i = 0; i < L; ++i) a[i] = __ldcs(pv + i * kRBlock);
#pragma unroll
    for (int i = 0; i < L; ++i) {
      V q = a[i];
      if constexpr (REF) q = __ldg(rv + i * kRBlock);
#pragma unroll
      for (int k = 0; k < W; ++k) f(vget(a[i], k), vget(q, k));
    }
  } else {                                             // a member smaller than a chunk
    for (uint64_t x = beg + threadIdx.x; x < N; x += blockDim.x) f(p[x], REF ? r[x] : p[x]);
  }
}

// partial[member][chunk] = sum over the chunk of conj(ref_i) psi_i.  Bound by
// HBM (the members; the reference stays in L2) and by the FP64 adds of the block
// sums (20 warp instructions of 64 cycles a block), so from 20 qubits on a block
// takes four rounds of 4096 amplitudes (chunk_rounds), a thread's sums of 16
// products added up in FP64 between rounds.  64 members of 2^20 complex64
// amplitudes, the call with its read-back: 209 -> 123 us, half of it the wide loads
// (two floats between rounds took 119, and were 48 bits with FP32's exponents).
template <typename R>
__global__ void __launch_bounds__(kRBlock) k_dot_partials(const cplx<R>* __restrict__ psi,
                                                          const cplx<R>* __restrict__ ref, int n,
                                                          int chunks, int rounds, double* partials) {
  const int c = blockIdx.x, b = blockIdx.y;
  const uint64_t N = 1ull << n;
  double sre = 0.0, sim = 0.0;
  for (int k = 0; k < rounds; ++k) {
    R re = 0, im = 0;
    chunk_each<R, true>(psi + (uint64_t)b * N, ref, ((uint64_t)c * rounds + k) * kChunk, N, [&](cplx<R> a, cplx<R> r) {
      re += r.x * a.x + r.y * a.y;
      im += r.x * a.y - r.y * a.x;
    });
    sre += (double)re;
    sim += (double)im;
  }
  const double2 s = block_sum2(sre, sim);
  if (threadIdx.x == 0) {
    partials[2 * ((uint64_t)b * chunks + c)] = s.x;
    partials[2 * ((uint64_t)b * chunks + c) + 1] = s.y;
  }
}

// partial[member][chunk] = sum |psi_i|^2 (stored in the .x slot)
template <typename R>
__global__ void __launch_bounds__(kRBlock) k_norm_partials(const cplx<R>* __restrict__ psi, int n,
                                                           int chunks, int rounds, double* partials) {
  const int c = blockIdx.x, b = blockIdx.y;
  const uint64_t N = 1ull << n;
  double sum = 0.0;
  for (int k = 0; k < rounds; ++k) {
    R s = 0;
    chunk_each<R, false>(psi + (uint64_t)b * N, psi, ((uint64_t)c * rounds + k) * kChunk, N,
                         [&](cplx<R> a, cplx<R>) { s += a.x * a.x + a.y * a.y; });
    sum += (double)s;
  }
  const double2 t = block_sum2(sum, 0.0);
  if (threadIdx.x == 0) {
    partials[2 * ((uint64_t)b * chunks + c)] = t.x;
    partials[2 * ((uint64_t)b * chunks + c) + 1] = 0.0;
  }
}

// v_b = |sum_c partial|^2 (mode 0) or sum_c partial.x (mode 1); out[g] =
// v_{g group} + ... + v_{g group + group - 1} in order (group = 1: out[b] =
// v_b).  WIDE = 0: one warp per output, lane l adds chunks l, l + 32, ... in
// order and the lanes meet in a fixed shuffle tree.  WIDE = 1: one block per
// output, its 8 warps shared out over the members of the group (8 / group
// warps each, at least one) and a member's warps taking its chunks in turn;
// their sums are added in warp order.  Either order is fixed by the shape.
// The kernel is a chain of dependent loads, so the wide form is taken when an
// output has more than 64 partials: one output of 16384 (a 14-qubit density
// matrix) 247 -> 24 us, 40 of 4096 (fused passes at 22 qubits) 30 -> 10 us; with
// fewer the narrow form starts fewer blocks and is as fast (4 us either way).
template <int WIDE>
__global__ void __launch_bounds__(256) k_finalize(const double* __restrict__ partials, int members, int chunks, int mode,
                                                  int group, double* __restrict__ out) {
  const double2* part = reinterpret_cast<const double2*>(partials);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int outs = members / group;
  auto strided = [&](const double2* pb, int first, int step) {
    double2 a[4] = {};
    int c = first;
    for (; c + 3 * step < chunks; c += 4 * step) {
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const double2 v = pb[c + k * step];
        a[k].x += v.x;
        a[k].y += v.y;
      }
    }
    for (; c < chunks; c += step) { const double2 v = pb[c]; a[0].x += v.x; a[0].y += v.y; }
    return make_double2(warp_sum((a[0].x + a[1].x) + (a[2].x + a[3].x)), warp_sum((a[0].y + a[1].y) + (a[2].y + a[3].y)));
  };
  if constexpr (WIDE == 0) {
    const int warps = (int)((gridDim.x * blockDim.x) >> 5);
    for (int g = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5); g < outs; g += warps) {
      double s = 0.0;
      for (int b = g * group; b < (g + 1) * group; ++b) {
        const double2 v = strided(part + (uint64_t)b * chunks, lane, 32);
        s += mode == 0 ? v.x * v.x + v.y * v.y : v.x;
      }
      if (lane == 0) out[g] = s;
    }
  } else {
    __shared__ double2 ws[8];
    const int per = group >= 8 ? 1 : 8 / group;          // warps per member
    const int at_once = 8 / per;                         // members summed side by side
    for (int g = blockIdx.x; g < outs; g += gridDim.x) {
      double s = 0.0;
      for (int b0 = 0; b0 < group; b0 += at_once) {
        const int b = b0 + warp / per;
        double2 v = make_double2(0.0, 0.0);
        if (b < group && warp < per * at_once)
          v = strided(part + ((uint64_t)g * group + b) * chunks, (warp % per) * 32 + lane, 32 * per);
        if (lane == 0) ws[warp] = v;
        __syncthreads();
        for (int k = 0; k < at_once && b0 + k < group; ++k) {
          double re = 0.0, im = 0.0;
          for (int q = 0; q < per; ++q) { re += ws[k * per + q].x; im += ws[k * per + q].y; }
          s += mode == 0 ? re * re + im * im : re;
        }
        __syncthreads();
      }
      if (threadIdx.x == 0) out[g] = s;
    }
  }
}

template <typename R>
__global__ void k_basis_prob(const cplx<R>* psi, int n, int members, uint64_t x, int group, double* out) {
  const int outs = members / group;
  for (int g = blockIdx.x * blockDim.x + threadIdx.x; g < outs; g += gridDim.x * blockDim.x) {
    double s = 0.0;
    for (int b = g * group; b < (g + 1) * group; ++b) {
      const cplx<R> a = psi[((uint64_t)b << n) + x];
      s += (double)a.x * a.x + (double)a.y * a.y;
    }
    out[g] = s;
  }
}

// tr(rho): sum_i Re rho[i][i] at vec index i * (2^n + 1)
template <typename R>
__global__ void __launch_bounds__(kRBlock) k_dm_trace_partials(const cplx<R>* rho, int n, int chunks,
                                                               int chunk, double* partials) {
  const uint64_t N = 1ull << n;
  const uint64_t beg = (uint64_t)blockIdx.x * chunk;
  double s = 0.0;
  for (int i = threadIdx.x; i < chunk; i += blockDim.x) {
    const uint64_t x = beg + i;
    if (x < N) s += (double)rho[x * (N + 1)].x;
  }
  const double2 t = block_sum2(s, 0.0);
  if (threadIdx.x == 0) { partials[2 * blockIdx.x] = t.x; partials[2 * blockIdx.x + 1] = 0.0; }
}

// <phi|rho|phi> = sum_i conj(phi_i) sum_j rho[i][j] phi_j, one block per row.
// HERM (an exactly Hermitian rho): the entries right of the diagonal only,
// their real part counted twice, 2 Re sum_{i<j}, plus the real diagonal; the
// part of a row that is summed starts at i, so blocks take rows from both
// ends in turn.  Bound by the FP64 pipe in complex128, four multiply-adds an
// entry (14 qubits 2.99 -> 0.99 ms for half the entries).
// complex64: the products and their sum in three floats (Sum3), phi scaled by
// 2^100 so that of the remainders only what is below 2^-249 is lost.  A row whose sum
// leaves FP32's range, or is so small (2^-172) that those could matter, is summed
// again in FP64: the result carries FP64's bits whatever the magnitudes (a row all
// of whose products are below 2^-249 is zero).  13 qubits, the call with its
// read-back: 1.44 ms with FP64 sums over the whole matrix, 0.18 so; two floats
// (48 bits) took 0.14.
constexpr float kExpectScale = 0x1p100f;
template <typename R, bool HERM>
__global__ void __launch_bounds__(kRBlock) k_dm_expect_rows(const cplx<R>* __restrict__ rho,
                                                            const cplx<R>* __restrict__ phi, int n,
                                                            double* partials) {
  const uint64_t N = 1ull << n;
  const uint64_t bi = blockIdx.x;
  const uint64_t i = HERM ? ((bi & 1) ? N - 1 - (bi >> 1) : bi >> 1) : bi;
  const cplx<R>* row = rho + i * N;
  // whole aligned steps of the block from the one that holds column i + 1
  const uint64_t j0 = HERM ? ((i + 1) & ~(uint64_t)(kRBlock - 1)) : 0;
  auto each = [&](auto&& f) {
#pragma unroll 4
    for (uint64_t j = j0 + threadIdx.x; j < N; j += kRBlock) {
      if (HERM && j <= i) continue;
      f(row[j], phi[j]);
    }
  };
  auto in64 = [&]() {
    double re = 0.0, im = 0.0;
    each([&](cplx<R> a, cplx<R> f) {
      re = fma((double)a.x, (double)f.x, re);
      re = fma(-(double)a.y, (double)f.y, re);
      im = fma((double)a.x, (double)f.y, im);
      im = fma((double)a.y, (double)f.x, im);
    });
    return block_sum2(re, im);
  };
  double2 v;
  if constexpr (sizeof(R) == 8) {
    v = in64();
  } else {
    Sum3 re, im;
    bool any = false;                    // a product that is not zero
    each([&](cplx<R> a, cplx<R> f) {
      f.x *= kExpectScale;
      f.y *= kExpectScale;
      re.add(a.x, f.x);
      re.add(-a.y, f.y);
      im.add(a.x, f.y);
      im.add(a.y, f.x);
      any |= re.s != 0.f || im.s != 0.f;
    });
    v = block_sum2(re.value(), im.value());
    any = __syncthreads_or(any);
    const double most = fmax(fabs(v.x), fabs(v.y));
    if (__syncthreads_or(threadIdx.x == 0 && any && !(most >= 0x1p-72 && most < 0x1p126))) {
      v = in64();
    } else {
      v.x *= 1.0 / (double)kExpectScale;
      v.y *= 1.0 / (double)kExpectScale;
    }
  }
  if (threadIdx.x == 0) {
    const cplx<R> f = phi[i];
    double r = (double)f.x * v.x + (double)f.y * v.y;                  // Re(conj(f) v)
    double m = (double)f.x * v.y - (double)f.y * v.x;
    if (HERM) {
      r = 2.0 * r + (double)row[i].x * ((double)f.x * f.x + (double)f.y * f.y);
      m = 0.0;
    }
    partials[2 * i] = r;
    partials[2 * i + 1] = m;
  }
}

template <typename R>
__global__ void k_convert_ref(const double* src, cplx<R>* dst, size_t count) {
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += (size_t)gridDim.x * blockDim.x)
    dst[i] = mk<R>((R)src[2 * i], (R)src[2 * i + 1]);
}

bool ensure_partials(qs_ctx* h, size_t doubles) {
  if (h->partials_cap >= doubles) return true;
  if (h->partials) cudaFreeAsync(h->partials, h->stream);
  h->partials = nullptr;
  h->partials_cap = 0;
  if (cudaMallocAsync((void**)&h->partials, doubles * sizeof(double), h->stream) != cudaSuccess) return false;
  h->partials_cap = doubles;
  return true;
}

// rounds of a block (a function of n alone: a member's sum does not depend on the
// batch; at 20 qubits one member still has 64 blocks) and blocks per member
int chunk_rounds(int n) { return n >= 20 ? 4 : 1; }
int chunk_count(int n) {
  const uint64_t N = 1ull << n, per = (uint64_t)kChunk * chunk_rounds(n);
  return (int)((N + per - 1) / per);
}

}  // namespace

cudaError_t launch_finalize(const double* partials, int members, int chunks, int mode, int group, double* out,
                            cudaStream_t s) {
  const int outs = members / group;
  if ((uint64_t)chunks * group > 64)                    // see k_finalize
    k_finalize<1><<<(unsigned)std::min(outs, 65535), 256, 0, s>>>(partials, members, chunks, mode, group, out);
  else
    k_finalize<0><<<(unsigned)std::max(1, std::min((outs + 7) / 8, 4096)), 256, 0, s>>>(partials, members, chunks, mode,
                                                                                      group, out);
  return cudaGetLastError();
}

cudaError_t launch_dot(qs_ctx* h, const void* psi, const void* ref, int n, int members,
                       int group, double* out) {
  const int chunks = chunk_count(n);
  if (!ensure_partials(h, (size_t)2 * chunks * members)) return cudaErrorMemoryAllocation;
  dim3 grid(chunks, members);
  if (h->dtype == QS_C64)
    k_dot_partials<float><<<grid, kRBlock, 0, h->stream>>>((const float2*)psi, (const float2*)ref, n, chunks, chunk_rounds(n), h->partials);
  else
    k_dot_partials<double><<<grid, kRBlock, 0, h->stream>>>((const double2*)psi, (const double2*)ref, n, chunks, chunk_rounds(n), h->partials);
  return launch_finalize(h->partials, members, chunks, 0, group, out, h->stream);
}

cudaError_t launch_norm(qs_ctx* h, const void* psi, int n, int members, int group, double* out) {
  const int chunks = chunk_count(n);
  if (!ensure_partials(h, (size_t)2 * chunks * members)) return cudaErrorMemoryAllocation;
  dim3 grid(chunks, members);
  if (h->dtype == QS_C64)
    k_norm_partials<float><<<grid, kRBlock, 0, h->stream>>>((const float2*)psi, n, chunks, chunk_rounds(n), h->partials);
  else
    k_norm_partials<double><<<grid, kRBlock, 0, h->stream>>>((const double2*)psi, n, chunks, chunk_rounds(n), h->partials);
  return launch_finalize(h->partials, members, chunks, 1, group, out, h->stream);
}

cudaError_t launch_basis_prob(qs_ctx* h, const void* psi, int n, int members, uint64_t x,
                              int group, double* out) {
  const unsigned g = (unsigned)((members / group + 255) / 256);
  if (h->dtype == QS_C64)
    k_basis_prob<float><<<g, 256, 0, h->stream>>>((const float2*)psi, n, members, x, group, out);
  else
    k_basis_prob<double><<<g, 256, 0, h->stream>>>((const double2*)psi, n, members, x, group, out);
  return cudaGetLastError();
}

cudaError_t launch_dm_trace(qs_ctx* h, const void* rho, int n, double* out) {
  const int chunks = (int)(((1ull << n) + kChunk - 1) / kChunk);
  if (!ensure_partials(h, (size_t)2 * chunks)) return cudaErrorMemoryAllocation;
  if (h->dtype == QS_C64)
    k_dm_trace_partials<float><<<chunks, kRBlock, 0, h->stream>>>((const float2*)rho, n, chunks, kChunk, h->partials);
  else
    k_dm_trace_partials<double><<<chunks, kRBlock, 0, h->stream>>>((const double2*)rho, n, chunks, kChunk, h->partials);
  return launch_finalize(h->partials, 1, chunks, 1, 1, out, h->stream);
}

cudaError_t launch_dm_expect(qs_ctx* h, const void* rho, const void* phi, int n, double* out) {
  const uint64_t N = 1ull << n;
  if (!ensure_partials(h, (size_t)2 * N)) return cudaErrorMemoryAllocation;
  const unsigned g = (unsigned)N;
  if (h->dtype == QS_C64) {
    auto *r = (const float2*)rho, *f = (const float2*)phi;
    if (h->hermitian) k_dm_expect_rows<float, true><<<g, kRBlock, 0, h->stream>>>(r, f, n, h->partials);
    else k_dm_expect_rows<float, false><<<g, kRBlock, 0, h->stream>>>(r, f, n, h->partials);
  } else {
    auto *r = (const double2*)rho, *f = (const double2*)phi;
    if (h->hermitian) k_dm_expect_rows<double, true><<<g, kRBlock, 0, h->stream>>>(r, f, n, h->partials);
    else k_dm_expect_rows<double, false><<<g, kRBlock, 0, h->stream>>>(r, f, n, h->partials);
  }
  // sum of N row partials: treat them as one member with N chunks, real part
  return launch_finalize(h->partials, 1, (int)N, 1, 1, out, h->stream);
}

cudaError_t launch_convert_ref(qs_ctx* h, const double* src, void* dst, size_t count) {
  const int g = (int)std::min<size_t>((count + 255) / 256, (size_t)num_sms() * 16);
  if (h->dtype == QS_C64) k_convert_ref<float><<<g, 256, 0, h->stream>>>(src, (float2*)dst, count);
  else k_convert_ref<double><<<g, 256, 0, h->stream>>>(src, (double2*)dst, count);
  return cudaGetLastError();
}

}  // namespace qs
