// Window sweeps of a Hermitian density matrix (Sec. 3): a run of one-qubit
// channels on a few qubits and of diagonal channels on any, applied with one read
// and one write of rho.
//
// rho is Hermitian and every channel keeps it so, so only tiles on and above the
// diagonal are read and computed; a tile above it is also written, conjugated and
// transposed, over its mirror image.  A tile is the block of rho whose row and
// column indices run over the same 64 values: the window's qubits and enough of
// the lowest qubits that every row of the tile is made of whole 32-byte sectors,
// in both orientations.
//
// One channel at a time costs a read of half of rho and a write of all of it (27
// sweeps for the 14-qubit QFT), which bounds complex64; in complex128 the FP64
// pipe does (2 lanes a clock and SM on GB300), and waited for memory between the
// short phases of a sweep.  With the tile in shared memory a window of w qubits
// and the diagonal channels between them are one sweep, and a noisy Hadamard
// takes 20 FP64 instructions for 4 entries instead of 32: its superoperator
// acts on the sums and differences of the 2 x 2 block.  Each diagonal run's factors
// (see k_dm_diag_block_herm) are applied to the four entries while they are in
// registers.  Measured, QFT and nothing else: 14 qubits complex128 67.5 -> 41.5 ms
// in 3 sweeps (a channel and its diagonal run 2.96 ms; the FP64 pipe alone would
// take 2.04), 13 qubits complex64 3.54 -> 1.07 ms in 4; relaxation of 13 qubits,
// complex64, 1.17 -> 0.84 ms in 4 sweeps.  A complex64 sweep with little
// arithmetic takes 210 us for 0.8 GB (0.57 of HBM): 32-byte rows keep the L1's
// request rate busy.
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>

#include "internal.cuh"

namespace qs {

namespace {

constexpr int kSide = 6;                 // log2 of a tile's side
constexpr int kS = 1 << kSide;
constexpr int kPitch = kS + 1;
constexpr int kDmThreads = 256;
constexpr int kDmOps = kDmWindowOps;
constexpr uint32_t kTrivial = 1u << 31;  // mask flag: factor 1, no noisy gate active

template <typename R> struct DmOp {
  int bit;                               // tile bit of the channel's qubit, -1: none
  int diag;                              // index of the diagonal run that follows, -1: none
  int form;                              // kHad: h, g, h2; kRelax: h = gamma, g = keep, h2 = c; kGeneral: S
  R h, g, h2;
  R S[16];
};
enum : int { kGeneral = 0, kHad = 1, kRelax = 2 };
template <typename R> struct DmDiag {
  const cplx<R>* u;
  const uint32_t* mask;
  R q[33];
};
template <typename R> struct DmArgs {
  int n, nops, ndiag;
  int pos[kSide];                        // qubits of the tile, ascending
  DmOp<R> ops[kDmOps];
  DmDiag<R> diag[kDmOps];
};

__device__ __forceinline__ uint32_t insert0(uint32_t v, int s) { return ((v >> s) << (s + 1)) | (v & ((1u << s) - 1)); }

// shared memory: the tile, then per diagonal run of the tile's 64 rows and 64
// columns the factor with the other index trivial, u and the mask, and the powers
// of sqrt(P)
template <typename R> __host__ __device__ constexpr size_t dm_tile_bytes() { return (size_t)kS * kPitch * sizeof(cplx<R>); }
constexpr int kPowers = 36;              // q^0 .. q^32, padded
template <typename R> __host__ __device__ constexpr size_t dm_diag_bytes() {
  return (size_t)2 * kS * (2 * sizeof(cplx<R>) + sizeof(uint32_t)) + kPowers * sizeof(R);
}

template <typename R>
__global__ void __launch_bounds__(kDmThreads) k_dm_window(cplx<R>* __restrict__ rho, const __grid_constant__ DmArgs<R> A) {
  using C = cplx<R>;
  extern __shared__ __align__(16) unsigned char dm_sm[];
  C* tile = reinterpret_cast<C*>(dm_sm);
  unsigned char* tabs = dm_sm + dm_tile_bytes<R>();
  __shared__ uint32_t off[kS];
  const int tid = threadIdx.x;
  const uint64_t N = 1ull << A.n;
  const uint32_t T = 1u << (A.n - kSide);
  const uint32_t bx = blockIdx.x / T, by = blockIdx.x % T;
  if (bx > by) return;
  // outer row and column indices: the bits outside the tile
  uint32_t x0 = bx, y0 = by;
#pragma unroll
  for (int k = 0; k < kSide; ++k) {
    x0 = insert0(x0, A.pos[k]);
    y0 = insert0(y0, A.pos[k]);
  }
  if (tid < kS) {
    uint32_t o = 0;
#pragma unroll
    for (int k = 0; k < kSide; ++k) o |= (uint32_t)((tid >> k) & 1) << A.pos[k];
    off[tid] = o;
  }
  __syncthreads();
  constexpr int kPerThread = kS * kS / kDmThreads;
  {
    const int c = tid % kS, r0 = tid / kS;
    const C* src = rho + y0 + off[c];
    C v[kPerThread];
#pragma unroll
    for (int k = 0; k < kPerThread; ++k)
      v[k] = src[(uint64_t)(x0 + off[r0 + k * (kDmThreads / kS)]) * N];
    // the diagonal runs' factors for this tile's rows and columns
    for (int d = tid / (2 * kS); d < A.ndiag; d += kDmThreads / (2 * kS)) {
      const int i = tid % (2 * kS), j = i % kS;
      const uint32_t x = (i < kS ? x0 : y0) + off[j];
      C* f = reinterpret_cast<C*>(tabs + d * dm_diag_bytes<R>());
      C* u = f + 2 * kS;
      uint32_t* mk_ = reinterpret_cast<uint32_t*>(u + 2 * kS);
      C ux = A.diag[d].u[x];
      const uint32_t m = A.diag[d].mask[x];
      if (i >= kS) ux.y = -ux.y;                         // columns enter conjugated
      const R q = A.diag[d].q[__popc(m & ~kTrivial)];
      u[i] = ux;
      f[i] = mk<R>(ux.x * q, ux.y * q);
      mk_[i] = m;
      if (i < 33) reinterpret_cast<R*>(mk_ + 2 * kS)[i] = A.diag[d].q[i];
    }
#pragma unroll
    for (int k = 0; k < kPerThread; ++k) tile[(r0 + k * (kDmThreads / kS)) * kPitch + c] = v[k];
  }
  __syncthreads();

  for (int o = 0; o < A.nops; ++o) {
    const DmOp<R>& op = A.ops[o];
    const int d = op.diag;
    const C* f = reinterpret_cast<const C*>(tabs + (d < 0 ? 0 : d) * dm_diag_bytes<R>());
    const C* u = f + 2 * kS;
    const uint32_t* mk_ = reinterpret_cast<const uint32_t*>(u + 2 * kS);
    const R* qs_ = reinterpret_cast<const R*>(mk_ + 2 * kS);
    const int b = op.bit < 0 ? 0 : op.bit;
    const int bit = 1 << b;
    const int form = op.bit < 0 ? -1 : op.form;
    // rows r, r | bit of warp-uniform r; the lanes take 32 column pairs
    const int c0 = (int)insert0((uint32_t)(tid & 31), b), c1 = c0 | bit;
    uint32_t mc0 = kTrivial, mc1 = kTrivial;
    C fc0 = mk<R>(R(1), R(0)), fc1 = fc0, uc0 = fc0, uc1 = fc0;
    if (d >= 0) {
      mc0 = mk_[kS + c0];
      mc1 = mk_[kS + c1];
      fc0 = f[kS + c0];
      fc1 = f[kS + c1];
      uc0 = u[kS + c0];
      uc1 = u[kS + c1];
    }
    // the entry times its factor u(x) conj(u(y)) q^popcount(mask(x) ^ mask(y)),
    // formed only as far as row and column need
    auto apply = [&](C v, int r, uint32_t mr, uint32_t mc, C fc, C uc) {
      if (mr & kTrivial) return (mc & kTrivial) ? v : cmul(v, fc);
      if (mc & kTrivial) return cmul(v, f[r]);
      const C ur = u[r];
      const R q = qs_[__popc(mr ^ mc)];
      const C g = cmul(ur, uc);
      return cmul(v, mk<R>(g.x * q, g.y * q));
    };
#pragma unroll 2
    for (int g = tid >> 5; g < kS / 2; g += kDmThreads / 32) {
      const int r0 = (int)insert0((uint32_t)g, b), r1 = r0 | bit;
      C* p0 = tile + r0 * kPitch;
      C* p1 = tile + r1 * kPitch;
      C e00 = p0[c0], e01 = p0[c1], e10 = p1[c0], e11 = p1[c1];
      if (form == kHad) {
        // a' = h s + g x, d' = h s - g x, b' = g z - h2 y, c' = g z + h2 y with
        // s, z = a +- d and x, y = b +- c
        auto part = [&](R& a, R& bb, R& cc, R& dd) {
          const R s = a + dd, z = a - dd, x = bb + cc, y = bb - cc;
          const R hs = op.h * s, hy = op.h2 * y;
          a = fma(op.g, x, hs);
          dd = fma(-op.g, x, hs);
          bb = fma(op.g, z, -hy);
          cc = fma(op.g, z, hy);
        };
        part(e00.x, e01.x, e10.x, e11.x);
        part(e00.y, e01.y, e10.y, e11.y);
      } else if (form == kRelax) {
        // a += gamma d, d *= keep, b and c *= the coherence factor
        auto part = [&](R& a, R& bb, R& cc, R& dd) {
          a = fma(op.h, dd, a);
          dd *= op.g;
          bb *= op.h2;
          cc *= op.h2;
        };
        part(e00.x, e01.x, e10.x, e11.x);
        part(e00.y, e01.y, e10.y, e11.y);
      } else if (form == kGeneral) {
        auto part = [&](R& a, R& bb, R& cc, R& dd) {
          const R i0 = a, i1 = bb, i2 = cc, i3 = dd;
          auto row = [&](int q) {
            return fma(op.S[4 * q], i0, fma(op.S[4 * q + 1], i1, fma(op.S[4 * q + 2], i2, op.S[4 * q + 3] * i3)));
          };
          a = row(0);
          bb = row(1);
          cc = row(2);
          dd = row(3);
        };
        part(e00.x, e01.x, e10.x, e11.x);
        part(e00.y, e01.y, e10.y, e11.y);
      }
      if (d >= 0) {
        const uint32_t m0 = mk_[r0], m1 = mk_[r1];
        e00 = apply(e00, r0, m0, mc0, fc0, uc0);
        e01 = apply(e01, r0, m0, mc1, fc1, uc1);
        e10 = apply(e10, r1, m1, mc0, fc0, uc0);
        e11 = apply(e11, r1, m1, mc1, fc1, uc1);
      }
      p0[c0] = e00;
      p0[c1] = e01;
      p1[c0] = e10;
      p1[c1] = e11;
    }
    __syncthreads();
  }

  {
    const int c = tid % kS, r0 = tid / kS;
    C* dst = rho + y0 + off[c];
#pragma unroll
    for (int k = 0; k < kPerThread; ++k) {
      const int r = r0 + k * (kDmThreads / kS);
      // on the diagonal the entries below it are the conjugates of those above,
      // exactly (they were computed on their own)
      C v = tile[r * kPitch + c];
      if (bx == by && r > c) v = cconj(tile[c * kPitch + r]);
      if (bx == by && r == c) v.y = R(0);
      dst[(uint64_t)(x0 + off[r]) * N] = v;
    }
    if (bx == by) return;
    C* mir = rho + x0 + off[c];                          // the mirrored tile: row r of it is column r here
#pragma unroll
    for (int k = 0; k < kPerThread; ++k) {
      const int r = r0 + k * (kDmThreads / kS);
      mir[(uint64_t)(y0 + off[r]) * N] = cconj(tile[c * kPitch + r]);
    }
  }
}

template <typename R>
cudaError_t launch_r(qs_ctx* h, const DmWindowOp* ops, int nops) {
  DmArgs<R> A{};
  A.n = h->n;
  uint64_t win = 0;
  for (int i = 0; i < nops; ++i) if (ops[i].qubit >= 0) win |= 1ull << ops[i].qubit;
  for (int q = 0; __builtin_popcountll(win) < kSide; ++q) win |= 1ull << q;     // the lowest qubits fill the tile
  int np = 0;
  int bit_of[64];
  for (int q = 0; q < h->n; ++q) {
    bit_of[q] = np;
    if ((win >> q) & 1) A.pos[np++] = q;
  }
  for (int i = 0; i < nops; ++i) {
    const DmWindowOp& o = ops[i];
    DmOp<R>& d = A.ops[A.nops++];
    d.bit = o.qubit < 0 ? -1 : bit_of[o.qubit];
    d.diag = -1;
    if (o.qubit >= 0 && o.relax) {
      d.form = kRelax;
      d.h = (R)o.S[3];
      d.g = (R)o.S[15];
      d.h2 = (R)o.S[5];
    } else if (o.qubit >= 0) {
      const double* S = o.S;
      // [h g g h], [g -h2 h2 -g], [g h2 -h2 -g], [h -g -g h] up to rounding
      const double hh = 0.25 * (S[0] + S[3] + S[12] + S[15]), h2 = 0.25 * (-S[5] + S[6] + S[9] - S[10]);
      const double g = 0.125 * (S[1] + S[2] + S[4] - S[7] + S[8] - S[11] - S[13] - S[14]);
      const double form[16] = {hh, g, g, hh, g, -h2, h2, -g, g, h2, -h2, -g, hh, -g, -g, hh};
      bool had = true;
      for (int k = 0; k < 16; ++k) {
        had &= S[k] - form[k] <= 4e-16 && form[k] - S[k] <= 4e-16;
        d.S[k] = (R)S[k];
      }
      d.form = had ? kHad : kGeneral;
      d.h = (R)hh;
      d.g = (R)g;
      d.h2 = (R)h2;
    }
    if (o.mask) {
      d.diag = A.ndiag;
      DmDiag<R>& t = A.diag[A.ndiag++];
      t.u = static_cast<const cplx<R>*>(o.u);
      t.mask = o.mask;
      double q = 1.0;
      for (int k = 0; k <= 32; ++k, q *= o.q) t.q[k] = (R)q;
    }
  }
  const size_t sm = dm_tile_bytes<R>() + (size_t)A.ndiag * dm_diag_bytes<R>();
  const uint64_t T = 1ull << (h->n - kSide);
  k_dm_window<R><<<(unsigned)(T * T), kDmThreads, sm, h->stream>>>(static_cast<cplx<R>*>(h->state), A);
  return cudaGetLastError();
}

}  // namespace

// Window of a sweep: in complex64 four qubits and the two lowest (rows of 32
// bytes), in complex128 five and the lowest.  A tile is one block's work, 50 us in
// complex128: from 11 qubits on (528 tiles) every SM has some; a 10-qubit QFT
// would keep 136 SMs for two sweeps as long as its 19 single sweeps take.  In
// complex64 a tile takes under 10 us, less than the launches it replaces.
int dm_window_qubits(const qs_ctx* h) { return h->dtype == QS_C64 ? 4 : 5; }

bool dm_window_applicable(const qs_ctx* h) {
  return h->mode == QS_DENSITY && h->n >= (h->dtype == QS_C64 ? 8 : 11) && h->n <= 21;
}

cudaError_t dm_window_attributes(const qs_ctx* h) {
  static std::atomic<bool> done[2] = {false, false};
  const int which = h->dtype == QS_C64 ? 0 : 1;
  if (done[which].load()) return cudaSuccess;
  const size_t most = which == 0 ? dm_tile_bytes<float>() + kDmOps * dm_diag_bytes<float>()
                                 : dm_tile_bytes<double>() + kDmOps * dm_diag_bytes<double>();
  cudaError_t e = which == 0
      ? cudaFuncSetAttribute(k_dm_window<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most)
      : cudaFuncSetAttribute(k_dm_window<double>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
  if (e == cudaSuccess)
    e = which == 0 ? cudaFuncSetAttribute(k_dm_window<float>, cudaFuncAttributePreferredSharedMemoryCarveout, 100)
                   : cudaFuncSetAttribute(k_dm_window<double>, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
  if (e == cudaSuccess) done[which].store(true);
  return e;
}

cudaError_t launch_dm_window(qs_ctx* h, const DmWindowOp* ops, int nops) {
  return h->dtype == QS_C64 ? launch_r<float>(h, ops, nops) : launch_r<double>(h, ops, nops);
}

}  // namespace qs
