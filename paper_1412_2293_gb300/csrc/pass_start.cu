// The fused passes of a run from a start that is not in memory yet (a basis state
// or the maximally entangled state): the kernels of pass.cuh instantiated with
// START, in a translation unit of their own so the library's units compile in
// parallel.
#include "pass.cuh"

namespace qs {
namespace fused {

namespace {
// the kernels of one window width: low with W warps, high with tiles of 2^CB columns
template <typename R, int M, int W, int CB, int NB, int FULL, typename F>
cudaError_t each(F&& f) {
  cudaError_t e = f(k_pass_low<R, W, 1, 0, M, true>, low_smem<R, W, 1, M>(), 1);
  if (e == cudaSuccess) e = f(k_pass_high<R, CB, NB, false, 0, M, true>, high_smem<R, CB, NB, M>(), NB == 1 && M == kWin ? 2 : 1);
  if constexpr (FULL != 0) {
    if (e == cudaSuccess) e = f(k_pass_low<R, W, 1, FULL, M, true>, low_smem<R, W, 1, M>(), 1);
    if (e == cudaSuccess) e = f(k_pass_high<R, CB, NB, false, FULL, M, true>, high_smem<R, CB, NB, M>(), NB == 1 && M == kWin ? 2 : 1);
  }
  return e;
}

template <typename R, int M, int W, int CB, int NB, int FULL>
cudaError_t launch(cplx<R>* psi, const CUtensorMap& tmap, const PassArgs& A, bool high, bool full, int sms, cudaStream_t s) {
  using L = LowShape<W, 1, M>;
  using H = HighShape<CB, M>;
  auto grid = [](uint64_t units, uint64_t cap) { return (unsigned)(units < cap ? units : cap); };
  if (!high) {
    const unsigned g = grid(A.tiles, sms);
    const size_t sm = low_smem<R, W, 1, M>();
    if constexpr (FULL != 0) {
      if (full) {
        k_pass_low<R, W, 1, FULL, M, true><<<g, L::THREADS, sm, s>>>(psi, A);
        return cudaGetLastError();
      }
    }
    k_pass_low<R, W, 1, 0, M, true><<<g, L::THREADS, sm, s>>>(psi, A);
  } else {
    const unsigned g = grid(A.tiles, (uint64_t)sms * (NB == 1 && M == kWin ? 2 : 1));
    const size_t sm = high_smem<R, CB, NB, M>();
    if (A.n > 32) {                                      // 64-bit member-local offsets
      if constexpr (M == kWin) k_pass_high<R, CB, 2, true, 0, M, true><<<grid(A.tiles, sms), H::THREADS, high_smem<R, CB, 2, M>(), s>>>(psi, tmap, A);
      else return cudaErrorInvalidValue;
      return cudaGetLastError();
    }
    if constexpr (FULL != 0) {
      if (full) {
        k_pass_high<R, CB, NB, false, FULL, M, true><<<g, H::THREADS, sm, s>>>(psi, tmap, A);
        return cudaGetLastError();
      }
    }
    k_pass_high<R, CB, NB, false, 0, M, true><<<g, H::THREADS, sm, s>>>(psi, tmap, A);
  }
  return cudaGetLastError();
}
}  // namespace

template <>
cudaError_t launch_pass_start<float>(cplx<float>* psi, const CUtensorMap& tmap, const PassArgs& A, bool high, int m, int prog,
                                     int sms, cudaStream_t s) {
  if (m == 11) return launch<float, 11, 12, wide_colb(11), 1, wide_full_prog(11)>(psi, tmap, A, high, prog == wide_full_prog(11), sms, s);
  if (m == 12) return launch<float, 12, 12, wide_colb(12), 1, wide_full_prog(12)>(psi, tmap, A, high, prog == wide_full_prog(12), sms, s);
  return launch<float, kWin, 12, 3, 1, kQftProg>(psi, tmap, A, high, prog == kQftProg, sms, s);
}

template <>
cudaError_t launch_pass_start<double>(cplx<double>* psi, const CUtensorMap& tmap, const PassArgs& A, bool high, int, int,
                                      int sms, cudaStream_t s) {
  return launch<double, kWin, 8, 2, 2, 0>(psi, tmap, A, high, false, sms, s);
}

cudaError_t set_start_attrs(size_t esize) {
  auto f = [](auto kernel, size_t dyn, int blocks) { return set_pass_attrs(kernel, dyn, blocks); };
  if (esize != 8) {
    const cudaError_t e = each<double, kWin, 8, 2, 2, 0>(f);
    return e != cudaSuccess ? e : f(k_pass_high<double, 2, 2, true, 0, kWin, true>, high_smem<double, 2, 2>(), 1);
  }
  cudaError_t e = each<float, kWin, 12, 3, 1, kQftProg>(f);
  if (e == cudaSuccess) e = each<float, 11, 12, wide_colb(11), 1, wide_full_prog(11)>(f);
  if (e == cudaSuccess) e = each<float, 12, 12, wide_colb(12), 1, wide_full_prog(12)>(f);
  if (e == cudaSuccess) e = f(k_pass_high<float, 3, 2, true, 0, kWin, true>, high_smem<float, 3, 2>(), 1);
  return e;
}

}  // namespace fused
}  // namespace qs
