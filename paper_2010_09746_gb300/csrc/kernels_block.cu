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
// Two ways to bring the amplitudes in, chosen by the lowest target bit (see use_staged):
//  - direct: thread t's group is group t; for target bits >= 3 (8-byte elements) or >= 2 (16-byte)
//    the lanes of a warp cover the low bits, and every load and store moves whole sectors;
//  - staged: a warp takes the 2^(K+5) amplitudes over the target bits and the 5 lowest other
//    bits.  That index set holds the lowest storage bits, so the warp moves them in storage
//    order, 32 consecutive ranks per instruction, through a padded shared-memory buffer of its
//    own (no block barrier) from which each lane takes its group.
//
// What bounds it: HBM up to K = 4 for complex64 (64 FMA per amplitude against 16 bytes), the FMA
// pipe at K = 5; double-float arithmetic and the binary64 split / join for complex128.  Measured on
// a 27-qubit complex64 state: nine blocks (K = 2 .. 5, and one K = 6 on the tensor cores with its
// permutations) 36.8 -> 5.8 ms; ten 1- and 2-qubit gates on a 26-qubit complex128 state 5.56 -> 4.96 ms.
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
template <class A, int K>
struct BlockMat {
  typename A::mat_t u[1 << (2 * K)];
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
__device__ __forceinline__ typename A::reg_t block_row(const typename A::mat_t* u, const typename A::reg_t (&x)[1 << K]) {
  if constexpr (K == 1) {
    return A::mac2(u[0], x[0], u[1], x[1]);
  } else {
    typename A::reg_t acc;
    if constexpr (std::is_same<A, ADF>::value) acc = A::mul(u[0], x[0]);
    else acc = A::mac(A::zero(), u[0], x[0]);
#pragma unroll
    for (int c = 1; c < (1 << K); c++) acc = A::mac(acc, u[c], x[c]);
    return acc;
  }
}
template <int K>
struct RowBlock {   // rows computed between two turns of the row loop
  static constexpr int value = K <= 2 ? (1 << K) : 4;
};

template <class A, int K>
__global__ void __launch_bounds__(kThreads, K >= 4 ? 4 : 1) k_block_direct(typename A::store_t* __restrict__ psi,
                                                          const __grid_constant__ BlockArgs<K> a,
                                                          const __grid_constant__ BlockMat<A, K> m) {
  using R = typename A::reg_t;
  constexpr int D = 1 << K, RB = RowBlock<K>::value;
  for (uint64_t t = (uint64_t)blockIdx.x * kThreads + threadIdx.x; t < a.nwork; t += (uint64_t)gridDim.x * kThreads) {
    typename A::store_t* p = psi + (expand_bits(t, a.pos, a.nz) | a.ones);
    typename A::store_t v[D];
    R x[D];
#pragma unroll
    for (int r = 0; r < D; r++) v[r] = p[a.off[r]];
#pragma unroll
    for (int r = 0; r < D; r++) x[r] = A::from_store(v[r]);
#pragma unroll 1
    for (int r0 = 0; r0 < D; r0 += RB) {
      R y[RB];
#pragma unroll
      for (int q = 0; q < RB; q++) y[q] = block_row<A, K>(m.u + (r0 + q) * D, x);
#pragma unroll
      for (int q = 0; q < RB; q++) p[a.off[r0 + q]] = A::to_store(y[q]);
    }
  }
}

template <class A, int K>
__global__ void __launch_bounds__(kThreads, K >= 4 ? 4 : 1) k_block_staged(typename A::store_t* __restrict__ psi,
                                                          const __grid_constant__ BlockArgs<K> a,
                                                          const __grid_constant__ BlockMat<A, K> m) {
  using R = typename A::reg_t;
  using S = typename A::store_t;
  constexpr int D = 1 << K, RB = RowBlock<K>::value, SH = PadShift<S, K>::value;
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
        buf[lane_pad + a.row_pad[r0 + q]] = A::to_store(block_row<A, K>(m.u + (r0 + q) * D, x));
    }
    __syncwarp();
#pragma unroll
    for (int j = 0; j < D; j++) p[a.off[j]] = buf[32 * j + lane + ((32 * j + lane) >> SH)];
    __syncwarp();
  }
}

// direct below costs extra sectors and lines per access; staged costs a round trip through shared
// memory
template <class S>
bool use_staged(int lowest_target) {
  return lowest_target < (sizeof(S) == 16 ? 2 : 3);
}

template <class A, int K>
cudaError_t launch_block_t(void* psi, int n, const int* kq, uint64_t ctl, const double* u, cudaStream_t st) {
  using S = typename A::store_t;
  constexpr int D = 1 << K;
  BlockMat<A, K> m;
  for (int e = 0; e < D * D; e++) host_entry(u + 2 * e, &m.u[e]);
  BlockArgs<K> a{};
  uint64_t targets = 0;
  int low = 64;
  for (int b = 0; b < K; b++) {
    targets |= 1ull << kq[b];
    low = std::min(low, kq[b]);
  }
  uint64_t fixed = targets | ctl;
  const int nfree = n - __builtin_popcountll(fixed);
  const bool staged = use_staged<S>(low) && nfree >= 5;
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
  int sms = 0, dev = 0, per_sm = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess)
    e = staged ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_block_staged<A, K>, kThreads, 0)
               : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_block_direct<A, K>, kThreads, 0);
  if (e != cudaSuccess) return e;
  const uint64_t per_block = staged ? kWarps : kThreads;
  const uint64_t grid = std::min<uint64_t>((a.nwork + per_block - 1) / per_block, (uint64_t)sms * std::max(per_sm, 1));
  if (staged) k_block_staged<A, K><<<(unsigned)grid, kThreads, 0, st>>>((S*)psi, a, m);
  else k_block_direct<A, K><<<(unsigned)grid, kThreads, 0, st>>>((S*)psi, a, m);
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
      if constexpr (std::is_same<A, AF32>::value) return launch_block_t<A, 5>(psi, n, kq, ctl, u, st);
      break;
  }
  return cudaErrorInvalidValue;
}

}  // namespace

// Register blocks: up to 32 complex64 or 16 complex128 amplitudes per thread (more would not fit the
// registers), with at most 6 controls
bool block_supported(Policy pol, int k, uint64_t ctl) {
  return k >= 1 && k <= (pol == POL_F32 ? 5 : 4) && __builtin_popcountll(ctl) <= 6;
}

cudaError_t launch_block(Policy pol, void* psi, int n, int k, const int* kq, uint64_t ctl, const double* u,
                         cudaStream_t s) {
  switch (pol) {
    case POL_F32: return launch_block_k<AF32>(psi, n, k, kq, ctl, u, s);
    case POL_F64: return launch_block_k<AF64>(psi, n, k, kq, ctl, u, s);
    case POL_DF: return launch_block_k<ADF>(psi, n, k, kq, ctl, u, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace qs
