// K1 for general blocks: a dense 2^K x 2^K matrix (K = 1..5) on any K storage bits, one group
// of 2^K amplitudes per thread, held in registers.
//
// The matrix is a kernel parameter: its entries are constant-bank operands at uniform
// addresses, so the multiply-adds take no load from shared or global memory (with the matrix
// in global memory and one output row per thread, every multiply-add waited for a matrix load
// and a shared-memory load), and a call uploads nothing.  Each thread computes the rows of its group one
// block of rows at a time and stores every row as it is done: the inputs are in registers, so
// the update in place needs no second copy of the group.
//
// Two ways to bring the amplitudes in, chosen by the low target bits (see use_staged):
//  - direct: thread t's group is group t; where the lanes of a warp cover the low bits, every load and
//    store moves whole sectors;
//  - staged: a warp takes the 2^(K+5) amplitudes over the target bits and the 5 lowest other
//    bits.  That index set holds the lowest storage bits, so the warp moves them in storage
//    order, 32 consecutive ranks per instruction, through a padded shared-memory buffer of its
//    own (no block barrier) from which each lane takes its group (complex64, two to four qubits).
//
// What bounds it.  complex64: HBM up to K = 4 (64 FMA per amplitude against 16 bytes), the FMA pipe at
// K = 5.  Double-float: at K = 1, 2 the binary64 split / join and the bytes together, from K = 3 on the FMA
// pipe (44 * 2^K lane operations per amplitude: 56, 76 and 76 % of it at K = 3, 4, 5).  Measured on a 27-qubit complex64
// state: ten blocks (K = 2 .. 6, low and spread qubits, three of them on the tensor cores) 36.8 -> 5.0 ms,
// K = 4 on high bits 0.375 ms (5.74 TB/s), K = 5 0.72 ms (24 T FMA/s); complex128 at 26 qubits: K = 1 0.44 ms
// (4.8 TB/s), K = 2 0.54, K = 3 0.84, K = 4 1.52, K = 5 3.09 ms (21 ms with one output row per thread).
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <atomic>
#include <type_traits>

#include "arith.cuh"
#include "qs_internal.h"

namespace qs {

namespace {

constexpr int kThreads = 128;
constexpr int kWarps = kThreads / 32;

// what the kernel needs besides the matrix
template <int K>
struct BlockArgs {
  uint64_t nwork;             // groups (direct) or warp tiles (staged)
  uint64_t ones;              // control bits
  int nz;                     // fixed bits: targets, controls, and (staged) the lane bits
  int pos[16];                // their storage positions, ascending
  uint64_t off[1 << K];       // direct: storage offset of row r; staged: of transfer j (ranks 32 j ..)
  int lane_pos[5];            // staged: storage positions of ranks 0..4
  int lane_rank[5];           // staged: ranks of the lane bits of a group
  int row_pad[1 << K];        // staged: padded position of row r's rank
};
// the matrix, row-major
template <class A, int K>
struct BlockMat {
  typename A::mat_t u[1 << (2 * K)];
  __device__ __forceinline__ const typename A::mat_t& at(int i) const { return u[i]; }
  void set(int i, const double* z) { host_entry(z, &u[i]); }
};
// 1024 double-float entries of 32 bytes would be four bytes more than the kernel parameters may take
// (32764): 24 bytes each, the low parts once and their lane patterns made where they are used
template <>
struct BlockMat<ADFG, 5> {
  float4 h[1024];
  float2 l[1024];   // (-ur.lo, ui.lo)
  __device__ __forceinline__ dfm at(int i) const {
    const float2 v = l[i];
    dfm m;
    m.h = h[i];
    m.l = make_float4(v.x, v.x, -v.y, v.y);
    return m;
  }
  void set(int i, const double* z) {
    dfm m;
    host_entry(z, &m);
    h[i] = m.h;
    l[i] = make_float2(m.l.x, m.l.w);
  }
};

__device__ __forceinline__ uint64_t expand_bits(uint64_t t, const int* pos, int nz) {
  for (int k = 0; k < nz; k++) {
    const int p = pos[k];
    t = ((t >> p) << (p + 1)) | (t & ((1ull << p) - 1));
  }
  return t;
}

// padding of the staged buffer (elements): a lane's rank times the group size plus this spreads the
// lanes of one shared-memory phase over all banks
template <class S, int K>
struct PadShift {
  static constexpr int value = sizeof(S) == 16 ? (K > 3 ? K : 3) : (K > 4 ? K : 4);
};

// row r of the block on the inputs x
template <class A, int K>
__device__ __forceinline__ typename A::reg_t block_row(const BlockMat<A, K>& m, int r, const typename A::reg_t (&x)[1 << K]) {
  const int i = r << K;
  if constexpr (K == 1) {
    return A::mac2(m.at(i), x[0], m.at(i + 1), x[1]);
  } else {
    typename A::reg_t acc;
    if constexpr (std::is_base_of<ADF, A>::value) acc = A::mul(m.at(i), x[0]);
    else acc = A::mac(A::zero(), m.at(i), x[0]);
#pragma unroll
    for (int c = 1; c < (1 << K); c++) acc = A::mac(acc, m.at(i + c), x[c]);
    return acc;
  }
}
// How a kernel is compiled.  kRows: rows computed between two turns of the row loop (all: more code,
// nothing gained).  kCtas: CTAs per SM the registers are limited to.
//  - complex64 K = 4 needs the loads of 24 warps in flight (16 warps: 590 us against 375 on a 27-qubit
//    state), K = 5 holds 64 registers of inputs; fewer qubits are at the HBM rate as the compiler leaves them.
//    The staged K = 4 kernel would spill 80 bytes at 24 warps: it has a limit of its own, 20 warps
//    without spills (27 qubits, bits 0-3, us, at 4 / 5 / 6 CTAs: 505 / 465 / 495).
//  - double-float: a thread has long dependent chains before its first load and after its last, so
//    more warps pay, at K = 3 even with 16 bytes spilled.  26 qubits, us, left to the compiler (K = 4: 4 CTAs)
//    -> limited as here: K = 1 465 -> 444 (8: 470, 12: 472), K = 2 595 -> 540 (10: 549, 12: 566), K = 3
//    1004 -> 839 (7: 978, 8: 849, 10: 878), K = 4 1870 -> 1521 (3: 1880, 6: 1573).  K = 5 holds 128 registers
//    of inputs: 3090 at 3 CTAs, 3580 at 2.  Two rows at a time are 2 % better than four at K = 3, four 20 %
//    worse than two at K = 5.
//  - native FP64 is bound by its pipe.
template <class A, int K>
struct BlockShape {
  static constexpr int kRows = K <= 2 ? (1 << K) : 4;
  static constexpr int kCtas = K < 4 ? 1 : (K == 4 && sizeof(typename A::store_t) == 8 ? 6 : 4);
  static constexpr int kStagedCtas = K == 4 ? 5 : kCtas;
};
template <int K>
struct BlockShape<ADFG, K> {
  static constexpr int kRows = K == 2 ? 4 : 2;
  static constexpr int kCtas = K == 1 ? 16 : K == 2 ? 8 : K == 3 ? 9 : K == 4 ? 5 : 3;
};

// kPair (complex64): storage bit 0 is target 0 of the block (the launcher orders the targets), so rows r and
// r + 1 of a group are neighbours and move as 16 bytes
template <class A, int K, bool kPair>
__global__ void __launch_bounds__(kThreads, BlockShape<A, K>::kCtas)
    k_block_direct(typename A::store_t* __restrict__ psi, const __grid_constant__ BlockArgs<K> a,
                   const __grid_constant__ BlockMat<A, K> m) {
  using R = typename A::reg_t;
  constexpr int D = 1 << K, RB = BlockShape<A, K>::kRows;
  for (uint64_t t = (uint64_t)blockIdx.x * kThreads + threadIdx.x; t < a.nwork; t += (uint64_t)gridDim.x * kThreads) {
    typename A::store_t* p = psi + (expand_bits(t, a.pos, a.nz) | a.ones);
    R x[D];
    if constexpr (kPair) {
      float4 v[D / 2];
#pragma unroll
      for (int r = 0; r < D; r += 2) v[r / 2] = *reinterpret_cast<const float4*>(p + a.off[r]);
#pragma unroll
      for (int r = 0; r < D; r += 2) {
        x[r] = make_float2(v[r / 2].x, v[r / 2].y);
        x[r + 1] = make_float2(v[r / 2].z, v[r / 2].w);
      }
    } else {
      typename A::store_t v[D];
#pragma unroll
      for (int r = 0; r < D; r++) v[r] = p[a.off[r]];
#pragma unroll
      for (int r = 0; r < D; r++) x[r] = A::from_store(v[r]);
    }
#pragma unroll 1
    for (int r0 = 0; r0 < D; r0 += RB) {
      R y[RB];
#pragma unroll
      for (int q = 0; q < RB; q++) y[q] = block_row<A, K>(m, r0 + q, x);
      if constexpr (kPair) {
#pragma unroll
        for (int q = 0; q < RB; q += 2)
          *reinterpret_cast<float4*>(p + a.off[r0 + q]) = make_float4(y[q].x, y[q].y, y[q + 1].x, y[q + 1].y);
      } else {
#pragma unroll
        for (int q = 0; q < RB; q++) p[a.off[r0 + q]] = A::to_store(y[q]);
      }
    }
  }
}

template <class A, int K>
__global__ void __launch_bounds__(kThreads, BlockShape<A, K>::kStagedCtas)
    k_block_staged(typename A::store_t* __restrict__ psi, const __grid_constant__ BlockArgs<K> a,
                   const __grid_constant__ BlockMat<A, K> m) {
  using R = typename A::reg_t;
  using S = typename A::store_t;
  constexpr int D = 1 << K, RB = BlockShape<A, K>::kRows, SH = PadShift<S, K>::value;
  constexpr int kBuf = (32 << K) + ((32 << K) >> SH);
  __shared__ S bufs[kWarps][kBuf];
  S* buf = bufs[threadIdx.x >> 5];
  const int lane = threadIdx.x & 31;
  uint64_t lane_off = 0;   // this lane's element within a transfer
  int lane_pad = 0;        // padded position of this lane's group
#pragma unroll
  for (int b = 0; b < 5; b++)
    if ((lane >> b) & 1) {
      lane_off |= 1ull << a.lane_pos[b];
      const int e = 1 << a.lane_rank[b];
      lane_pad += e + (e >> SH);
    }
  const uint64_t nw = (uint64_t)gridDim.x * kWarps;
  for (uint64_t t = (uint64_t)blockIdx.x * kWarps + (threadIdx.x >> 5); t < a.nwork; t += nw) {
    S* p = psi + (expand_bits(t, a.pos, a.nz) | a.ones | lane_off);
    S v[D];
#pragma unroll
    for (int j = 0; j < D; j++) v[j] = p[a.off[j]];
#pragma unroll
    for (int j = 0; j < D; j++) buf[32 * j + lane + ((32 * j + lane) >> SH)] = v[j];
    __syncwarp();
    R x[D];
#pragma unroll
    for (int r = 0; r < D; r++) x[r] = A::from_store(buf[lane_pad + a.row_pad[r]]);
    // a lane reads and then overwrites only its own group's places
#pragma unroll 1
    for (int r0 = 0; r0 < D; r0 += RB) {
#pragma unroll
      for (int q = 0; q < RB; q++)
        buf[lane_pad + a.row_pad[r0 + q]] = A::to_store(block_row<A, K>(m, r0 + q, x));
    }
    __syncwarp();
#pragma unroll
    for (int j = 0; j < D; j++) p[a.off[j]] = buf[32 * j + lane + ((32 * j + lane) >> SH)];
    __syncwarp();
  }
}

// Which way.  Direct moves 8 or 16 bytes per lane; the sectors and lines that one instruction leaves
// incomplete are completed by the next ones out of L1 and in L2, which is cheaper than the round trip
// through shared memory unless the lanes are spread far apart.  27 qubits complex64, us, staged / direct:
//   K = 2  bits 0 1: 332 / 365   1 2: 331 / 375   0 2: 331 / 336   2 3: 375 / 357   one low bit: 348 / 327
//   K = 3  bits 0 1 2: 374 / 353   1 2 3: 375 / 503   0 1 and a high one: 379 / 343   one low bit: 402 / 372
//   K = 4  bits 0-3: 465 / 568   1-4: 465 / 502   2-5: 492 / 373   0 1 and high ones: 495 / 420   one: 501 / 376
//          (the latter three staged at 24 warps)
//   K = 5  bits 0-4: 837 / 806   1-5: 839 / 752   one: 849 / 713
// complex128 (26 qubits): direct 357 against 441 at K = 1 on bit 0, 478 against 522 at K = 2 on bits 0 1, and equal
// or better beyond.
bool use_staged(bool c64, int K, uint64_t targets) {
  if (!c64) return false;
  if (K == 2) return (targets & ~7ull) == 0;
  return (K == 3 || K == 4) && (targets & 14ull) == 14ull;
}

template <class A, int K>
cudaError_t launch_block_t(void* psi, int n, const int* kq_in, uint64_t ctl, const double* u, cudaStream_t st) {
  using S = typename A::store_t;
  constexpr int D = 1 << K;
  constexpr bool kPairs = std::is_same<A, AF32>::value;
  // complex64: storage bit 0, where it is a target, becomes target 0 (exchanged with the first one, and the
  // matrix's rows and columns with it)
  int kq[K], at0 = -1;
  for (int b = 0; b < K; b++) {
    kq[b] = kq_in[b];
    if (kPairs && kq[b] == 0) at0 = b;
  }
  if (at0 > 0) std::swap(kq[0], kq[at0]);
  auto from = [&](int r) {   // the caller's row or column of ours
    if (at0 <= 0) return r;
    const int d = (r ^ (r >> at0)) & 1;
    return r ^ (d | (d << at0));
  };
  BlockMat<A, K> m;
  for (int r = 0; r < D; r++)
    for (int c = 0; c < D; c++) m.set(r * D + c, u + 2 * (from(r) * D + from(c)));
  BlockArgs<K> a{};
  uint64_t targets = 0;
  for (int b = 0; b < K; b++) targets |= 1ull << kq[b];
  uint64_t fixed = targets | ctl;
  const int nfree = n - __builtin_popcountll(fixed);
  constexpr bool kCanStage = kPairs && K >= 2 && K <= 4;
  const bool staged = use_staged(kPairs, K, targets) && nfree >= 5;
  a.ones = ctl;
  if (staged) {
    uint64_t lanes = 0, rest = ~fixed;
    for (int b = 0; b < 5; b++) {
      lanes |= rest & (0 - rest);
      rest &= rest - 1;
    }
    int rank_of[64], rank = 0;
    int where[K + 5];
    for (int b = 0; b < n; b++)
      if (((targets | lanes) >> b) & 1) {
        rank_of[b] = rank;
        where[rank++] = b;
      }
    for (int b = 0; b < 5; b++) a.lane_pos[b] = where[b];
    int lb = 0;
    for (int b = 0; b < n; b++)
      if ((lanes >> b) & 1) a.lane_rank[lb++] = rank_of[b];
    constexpr int SH = PadShift<S, K>::value;
    for (int r = 0; r < D; r++) {
      a.off[r] = 0;
      a.row_pad[r] = 0;
      for (int b = 0; b < K; b++)
        if ((r >> b) & 1) {
          a.off[r] |= 1ull << where[5 + b];
          const int e = 1 << rank_of[kq[b]];
          a.row_pad[r] += e + (e >> SH);
        }
    }
    fixed |= lanes;
    a.nwork = 1ull << (nfree - 5);
  } else {
    for (int r = 0; r < D; r++) {
      a.off[r] = 0;
      for (int b = 0; b < K; b++)
        if ((r >> b) & 1) a.off[r] |= 1ull << kq[b];
    }
    a.nwork = 1ull << nfree;
  }
  for (int b = 0; b < n; b++)
    if ((fixed >> b) & 1) a.pos[a.nz++] = b;
  // The paired form, with fewer registers at K = 2 and 3, takes the plain one's grid too: filled to its own
  // occupancy it is 3 to 6 % slower with one or two targets low and 5 % faster at K = 3 with bit 0 alone (27 qubits).
  int sms = 0, dev = 0, per_sm = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess)
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_block_direct<A, K, false>, kThreads, 0);
  if constexpr (kCanStage)
    if (e == cudaSuccess && staged) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_block_staged<A, K>, kThreads, 0);
  if (e != cudaSuccess) return e;
  const uint64_t per_block = staged ? kWarps : kThreads;
  const uint64_t grid = std::min<uint64_t>((a.nwork + per_block - 1) / per_block, (uint64_t)sms * std::max(per_sm, 1));
  if constexpr (kCanStage)
    if (staged) {
      k_block_staged<A, K><<<(unsigned)grid, kThreads, 0, st>>>((S*)psi, a, m);
      return cudaGetLastError();
    }
  if (kPairs && at0 >= 0) k_block_direct<A, K, kPairs><<<(unsigned)grid, kThreads, 0, st>>>((S*)psi, a, m);
  else k_block_direct<A, K, false><<<(unsigned)grid, kThreads, 0, st>>>((S*)psi, a, m);
  return cudaGetLastError();
}

template <class A>
cudaError_t launch_block_k(void* psi, int n, int k, const int* kq, uint64_t ctl, const double* u, cudaStream_t st) {
  switch (k) {
    case 1: return launch_block_t<A, 1>(psi, n, kq, ctl, u, st);
    case 2: return launch_block_t<A, 2>(psi, n, kq, ctl, u, st);
    case 3: return launch_block_t<A, 3>(psi, n, kq, ctl, u, st);
    case 4: return launch_block_t<A, 4>(psi, n, kq, ctl, u, st);
    case 5:
      if constexpr (!std::is_same<A, AF64>::value) return launch_block_t<A, 5>(psi, n, kq, ctl, u, st);
      break;
  }
  return cudaErrorInvalidValue;
}

}  // namespace

// Register blocks: up to 32 amplitudes per thread (16 in native FP64, whose pipe bounds the block at any
// layout), with at most 6 controls
bool block_supported(Policy pol, int k, uint64_t ctl) {
  return k >= 1 && k <= (pol == POL_F64 ? 4 : 5) && __builtin_popcountll(ctl) <= 6;
}

cudaError_t launch_block(Policy pol, void* psi, int n, int k, const int* kq, uint64_t ctl, const double* u,
                         cudaStream_t s) {
  switch (pol) {
    case POL_F32: return launch_block_k<AF32>(psi, n, k, kq, ctl, u, s);
    case POL_F64: return launch_block_k<AF64>(psi, n, k, kq, ctl, u, s);
    case POL_DF: return launch_block_k<ADFG>(psi, n, k, kq, ctl, u, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace qs
