// Qubit permutation (K3): PermuteQubits(sigma') as a bit-index transpose (Sec. 2, App. A).
//
// The vector stored under sigma is rewritten under sigma': out[j'] = in[j] where storage bit
// p of j' carries the logical qubit that sat at storage bit src_of[p] of j
// (src_of = sigma o sigma'^{-1}).  A pure move of whole elements: bit-exact.
//
// Each CTA moves tiles of 16 KiB through shared memory: the tile bits are the c lowest output bits
// and the input bits they come from, the c lowest input bits and the output bits they go to,
// and the lowest other input bits up to the tile size, so that HBM reads and writes both move
// 2^c-element (256-byte) contiguous runs.  The remaining bits enumerate tiles.  When storage
// bit 0 stays where it is, complex64 pairs of amplitudes move as 16-byte elements of a state with one
// bit less.
//
// Bound by HBM.  Every tile's loads are asynchronous copies (cp.async) into a ring of three buffers, two
// tiles ahead of the one being written, with one block barrier per tile: four CTAs keep 128 KiB of
// reads in flight per SM.  A thread's element offsets are its low bits' (fixed) and one constant per
// copy; a tile's base addresses come from one OR-reduction over the lanes of a warp, a lane per bit.
// The shared-memory position is XOR-swizzled with a period of the elements of one 128-byte phase, so that
// lanes that differ in any run of consecutive tile bits fall into different banks.
//
// Measured (two block barriers per tile and synchronous loads before): 28 qubits complex128, random and
// three-exchange permutations, 1.50 -> 1.33 ms each (6.45 TB/s, 95 % of the copy bandwidth); 27 qubits complex64
// 545 -> 329 us (6.53 TB/s); the single exchanges of Algorithm 1 at 26 qubits complex64 277 -> 173 us.
#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

#include "qs_internal.h"

namespace qs {

namespace {

constexpr int kPermThreads = 256;
constexpr int kPermTileBytes = 16 * 1024;
constexpr int kPermStages = 3;
constexpr int kPermCtasPerSm = 4;

template <class S>
struct PermShape {
  static constexpr int kElems = kPermTileBytes / (int)sizeof(S);     // 2048 / 1024
  static constexpr int kTileBits = sizeof(S) == 16 ? 10 : 11;
  static constexpr int kPerThread = kElems / kPermThreads;           // 8 / 4
  static constexpr int kLowBits = sizeof(S) == 16 ? 4 : 5;           // 256-byte runs
  static constexpr int kPhaseBits = sizeof(S) == 16 ? 3 : 4;         // elements of a 128-byte phase
};

template <class S>
struct PermArgs {
  int tb;                          // tile bits
  int nrest;                       // other bits
  int tin[11];                     // input storage bits of the tile, ascending
  int wk[11];                      // rank-th lowest output tile bit comes from tile bit wk[rank]
  int wp[11];                      // and sits at output position wp[rank]
  int8_t rin[32], rout[32];        // the other bits' input (ascending) and output positions
  // offsets of the tile-local indices 256 k (in input order) and of the output-ordered indices
  // 256 k, and the swizzled position of the tile-local index the latter read
  uint64_t in_hi[PermShape<S>::kPerThread], out_hi[PermShape<S>::kPerThread];
  int pos_hi[PermShape<S>::kPerThread];
};

// swizzled shared-memory position of tile-local index e: the bits above a phase folded into it (linear
// over XOR, so positions of disjoint bit sets combine by XOR)
template <class S>
__host__ __device__ __forceinline__ int swizzle(int e) {
  constexpr int B = PermShape<S>::kPhaseBits, M = (1 << B) - 1;
  return e ^ (((e >> B) ^ (e >> (2 * B)) ^ (e >> (3 * B))) & M);
}

template <class S>
__device__ __forceinline__ void copy_async(uint32_t dst, const S* src) {
  if constexpr (sizeof(S) == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void copy_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void copy_wait_all_but_one() { asm volatile("cp.async.wait_group 1;" ::: "memory"); }

// index bits of t deposited at per-lane positions p (one lane per bit): the same value on every lane
__device__ __forceinline__ uint64_t deposit(uint64_t t, int lane, int p, bool used) {
  const uint64_t v = (used && ((t >> lane) & 1ull)) ? (1ull << p) : 0ull;
  const uint32_t lo = __reduce_or_sync(0xffffffffu, (uint32_t)v);
  const uint32_t hi = __reduce_or_sync(0xffffffffu, (uint32_t)(v >> 32));
  return ((uint64_t)hi << 32) | lo;
}

template <class S>
__global__ void __launch_bounds__(kPermThreads, kPermCtasPerSm)
    k_permute(S* __restrict__ dst, const S* __restrict__ src, const __grid_constant__ PermArgs<S> a) {
  using P = PermShape<S>;
  extern __shared__ __align__(128) unsigned char smem[];
  S* ring = reinterpret_cast<S*>(smem);
  const int tid = threadIdx.x, lane = tid & 31;
  const int E = 1 << a.tb;
  // this thread's low bits: element tid of the tile in input order, and in output order
  uint64_t in_lo = 0, out_lo = 0;
  int r_lo = 0;
  for (int k = 0; k < 8 && k < a.tb; k++)
    if ((tid >> k) & 1) {
      in_lo |= 1ull << a.tin[k];
      out_lo |= 1ull << a.wp[k];
      r_lo |= 1 << a.wk[k];
    }
  const int wpos = swizzle<S>(tid), rpos = swizzle<S>(r_lo);
  const bool used = lane < a.nrest;
  const int my_in = a.rin[lane], my_out = a.rout[lane];
  const uint64_t ntiles = 1ull << a.nrest;
  auto load = [&](uint64_t t, int stage) {
    if (t < ntiles) {
      const S* p = src + (deposit(t, lane, my_in, used) | in_lo);
      const uint32_t d = (uint32_t)__cvta_generic_to_shared(ring + stage * P::kElems);
#pragma unroll
      for (int k = 0; k < P::kPerThread; k++)
        if (tid + kPermThreads * k < E)
          copy_async<S>(d + (uint32_t)sizeof(S) * (uint32_t)(wpos ^ swizzle<S>(kPermThreads * k)), p + a.in_hi[k]);
    }
    copy_commit();
  };
  uint64_t t = blockIdx.x;
  load(t, 0);
  load(t + gridDim.x, 1);
  int cur = 0;
  for (; t < ntiles; t += gridDim.x) {
    copy_wait_all_but_one();
    // tile t has landed, and every thread is done with the buffer before this one
    __syncthreads();
    const int ahead = cur >= 1 ? cur - 1 : kPermStages - 1;   // (cur + 2) mod 3
    load(t + 2 * (uint64_t)gridDim.x, ahead);
    const S* buf = ring + cur * P::kElems;
    S* q = dst + (deposit(t, lane, my_out, used) | out_lo);
    S v[P::kPerThread];
#pragma unroll
    for (int k = 0; k < P::kPerThread; k++)
      if (tid + kPermThreads * k < E) v[k] = buf[rpos ^ a.pos_hi[k]];
#pragma unroll
    for (int k = 0; k < P::kPerThread; k++)
      if (tid + kPermThreads * k < E) q[a.out_hi[k]] = v[k];
    cur = cur == kPermStages - 1 ? 0 : cur + 1;
  }
}

template <class S>
cudaError_t launch_permute_t(void* dst, const void* src, int n, const int* src_of, cudaStream_t s) {
  using P = PermShape<S>;
  // output bit p takes input bit src_of[p]; dst_of[input bit] = output bit
  int dst_of[kMaxQubits];
  for (int p = 0; p < n; p++) dst_of[src_of[p]] = p;
  const int c = P::kLowBits < n ? P::kLowBits : n;
  bool in_tile[kMaxQubits] = {};
  int count = 0;
  auto take = [&](int b) {
    count += !in_tile[b];
    in_tile[b] = true;
  };
  for (int p = 0; p < c; p++) {
    take(p);            // lowest input bits
    take(src_of[p]);    // input bits that become the lowest output bits
  }
  for (int b = 0; b < n && count < P::kTileBits; b++) take(b);
  PermArgs<S> a{};
  int tout[11];
  for (int b = 0; b < n; b++) {
    if (in_tile[b]) {
      a.tin[a.tb] = b;
      tout[a.tb] = dst_of[b];
      a.tb++;
    } else {
      a.rin[a.nrest] = (int8_t)b;
      a.rout[a.nrest] = (int8_t)dst_of[b];
      a.nrest++;
    }
  }
  // output tile bits in ascending output position
  int rank = 0;
  for (int p = 0; p < n; p++)
    for (int k = 0; k < a.tb; k++)
      if (tout[k] == p) {
        a.wk[rank] = k;
        a.wp[rank] = p;
        rank++;
      }
  for (int k = 0; k < P::kPerThread; k++) {
    int r = 0;
    for (int b = 8; b < a.tb; b++)
      if (((kPermThreads * k) >> b) & 1) {
        a.in_hi[k] |= 1ull << a.tin[b];
        a.out_hi[k] |= 1ull << a.wp[b];
        r |= 1 << a.wk[b];
      }
    a.pos_hi[k] = swizzle<S>(r);
  }
  constexpr size_t smem = (size_t)kPermStages * kPermTileBytes;   // 48 KiB: no opt-in needed
  int sms = 0, dev = 0;   // per device: the SM count of the current one
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  const uint64_t ntiles = 1ull << a.nrest;
  const uint64_t cap = (uint64_t)sms * kPermCtasPerSm;
  const uint64_t grid = ntiles < cap ? ntiles : cap;
  k_permute<S><<<(unsigned)grid, kPermThreads, smem, s>>>((S*)dst, (const S*)src, a);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_permute(void* dst, const void* src, int n, int store_bytes, const int* src_of, cudaStream_t s) {
  if (store_bytes == 16) return launch_permute_t<double2>(dst, src, n, src_of, s);
  if (n >= 2 && src_of[0] == 0) {   // pairs of amplitudes stay together
    int pair_of[kMaxQubits];
    for (int p = 1; p < n; p++) pair_of[p - 1] = src_of[p] - 1;
    return launch_permute_t<double2>(dst, src, n - 1, pair_of, s);
  }
  return launch_permute_t<float2>(dst, src, n, src_of, s);
}

}  // namespace qs
