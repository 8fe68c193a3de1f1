// Permutations between the natural layout and the solver layout (Section 5:
// the data of a chunk interleaved so that a warp reads one row of it as one
// contiguous run).  Internal to libhines.
#include <cuda_runtime.h>

#include <cstdint>

#include "kernels.h"
#include "unit_kernels.cuh"

namespace hines {
namespace {

// Unpacking chunk by chunk, a warp each (chunks do not depend on one another
// here).  A chunk's block is contiguous in the solver layout (row r: the r-th
// compartment from the distal end of every piece longer than r), and each of
// its pieces is one contiguous run in the plan's numbering.  The block arrives
// in shared memory in block order (R) by one bulk copy; each lane moves the
// slots of its own pieces, row by row (consecutive words of R), into piece
// order (C: one row of kPitch words per piece, kPitch odd); half-warps then
// write each piece's run to the natural layout (consecutive words of C).
// Neither side conflicts on shared-memory banks, and every global write is a
// contiguous run, as the solves write x.  kMapped: the plan's numbering is not
// the caller's (re-rooted plans), so the caller's index of every slot comes
// from the plan's slot map.  Latency bounds a chunk (block, then its runs), so
// as many warps as shared memory holds work at once.  (As a visit of the
// solves' task driver it walked every task twice, in two launches: 249 us for
// 21M compartments of 8 bytes; a warp
// per chunk 103 us, with the next chunk's metadata on its way 93 us; re-rooted
// plan 540, now 223 us.)
//
// (Packing stays slot by slot: a chunk-wise gather measured slower than the
// plain kernel below, 1.02 against 0.66 ms per FP32 array of the full
// uneven population, which reads scattered but writes contiguously.)
template <typename W, int P>
struct Unpack {
  using G = Geo<P>;
  static constexpr int kPitch = kL + 1;
  static constexpr int kRowBytes = (G::kSlots * (int)sizeof(W) + 15) / 16 * 16;          // R (holds a padded block)
  static constexpr int kColBytes = (G::kChunk * kPitch * (int)sizeof(W) + 15) / 16 * 16;  // C
  static constexpr int kTab = kRowBytes + kColBytes;                                     // the block's row offsets
  static constexpr int kWarpBytes = kTab + 96;
  static constexpr int kWarps = 4;
  using Bulk = BulkStage<kTab + 80>;
};

template <typename W, int P, bool kMapped>
__global__ void __launch_bounds__(32 * Unpack<W, P>::kWarps)
    k_unpack(DevPlan Pl, const W* __restrict__ src, W* __restrict__ dst, const int64_t* __restrict__ map) {
  using U = Unpack<W, P>;
  extern __shared__ __align__(16) unsigned char smem[];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  unsigned char* buf = smem + w * U::kWarpBytes;
  int* tab = reinterpret_cast<int*>(buf + U::kTab);
  const W* sr = reinterpret_cast<const W*>(buf);
  W* sc = reinterpret_cast<W*>(buf + U::kRowBytes);
  if (lane == 0) U::Bulk::init(buf);
  __syncwarp();
  // a chunk's metadata is loaded while the chunk before it is moved
  const int step = gridDim.x * U::kWarps;
  int n_next = 0;
  auto load = [&](int k) {
    int c0 = 0;
    n_next = 0;
    if (k < Pl.n_chunks) {
      c0 = __ldg(Pl.chunk_pos + k);
      n_next = __ldg(Pl.chunk_pos + k + 1) - c0;
    }
    return load_meta<false, P>(Pl, c0, n_next, lane, true);
  };
  int k = blockIdx.x * U::kWarps + w;
  RawMeta<false, P> r = load(k);
  for (; k < Pl.n_chunks; k += step) {
    const Meta<P> m = unpack_meta(r);
    const int n = n_next;
    build_row_table<P>(m.L, lane, tab);
    // the block with its padding: blocks start on multiples of 4 slots, so
    // this is the distance to the next block (whole 16-byte words)
    U::Bulk::template issue<1>(buf, lane, (unsigned)(((tab[kL] + 3) & ~3) * (int)sizeof(W)), buf, src + m.blk);
    r = load(k + step);
    U::Bulk::wait(Pl, buf, lane);
    for (int r = 0; r < m.L; ++r) {
      const int t = m.L - 1 - r;  // distance from the proximal end (pieces of a pair aligned there)
#pragma unroll
      for (int h = 0; h < P; ++h) {
        const int i = P * lane + h;
        if (t < m.p[h].len) sc[i * U::kPitch + t] = sr[tab[r] + i];
      }
    }
    __syncwarp();
    for_chunk_elements(m, n, lane, [&](int i, int t, int row, long long g) {
      const W v = sc[i * U::kPitch + t];
      if constexpr (kMapped) {
        const long long c = __ldg(map + m.blk + tab[row] + i);
        if (c >= 0) dst[c] = v;
      } else {
        dst[g] = v;
      }
    });
    __syncwarp();
  }
}

template <typename W, int P, bool kMapped>
cudaError_t unpack_by_chunks(const DevPlan& Pd, const W* pk, W* nat, cudaStream_t s) {
  using U = Unpack<W, P>;
  const int smem = U::kWarps * U::kWarpBytes;
  cudaError_t e = cudaFuncSetAttribute(k_unpack<W, P, kMapped>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  int per_sm = 0;
  if (e == cudaSuccess)
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_unpack<W, P, kMapped>, 32 * U::kWarps, smem);
  if (e != cudaSuccess) return e;
  const int need = (Pd.n_chunks + U::kWarps - 1) / U::kWarps, most = Pd.sms * (per_sm > 0 ? per_sm : 1);
  k_unpack<W, P, kMapped><<<need < most ? need : most, 32 * U::kWarps, smem, s>>>(Pd, pk, nat, Pd.pk_perm);
  return cudaGetLastError();
}

template <typename W>
cudaError_t unpack(const DevPlan& Pd, const void* packed, void* natural, cudaStream_t s) {
  const bool mapped = Pd.pk_edge != Pd.pk_perm;  // re-rooted: the plan's numbering is its own
  const W* pk = static_cast<const W*>(packed);
  W* nat = static_cast<W*>(natural);
  if (Pd.per_lane == 2)
    return mapped ? unpack_by_chunks<W, 2, true>(Pd, pk, nat, s) : unpack_by_chunks<W, 2, false>(Pd, pk, nat, s);
  return mapped ? unpack_by_chunks<W, 1, true>(Pd, pk, nat, s) : unpack_by_chunks<W, 1, false>(Pd, pk, nat, s);
}

// packed[p] = natural[perm[p]]; padding slots (perm -1) are set to zero.
template <typename W>
__global__ void k_pack(const int64_t* __restrict__ perm, int64_t n_packed, const W* __restrict__ nat,
                       W* __restrict__ pk) {
  for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < n_packed; p += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = perm[p];
    pk[p] = i >= 0 ? nat[i] : W(0);
  }
}

int blocks_for(int64_t n) {
  const int64_t b = (n + 255) / 256;
  return (int)(b < 4096 ? (b > 0 ? b : 1) : 4096);
}

}  // namespace

cudaError_t launch_pack(const DevPlan& P, int elem_bytes, const void* natural, void* packed, cudaStream_t s,
                        bool coupling) {
  if (P.n_packed == 0) return cudaSuccess;
  const int64_t* perm = coupling ? P.pk_edge : P.pk_perm;
  if (elem_bytes == 8)
    k_pack<uint64_t><<<blocks_for(P.n_packed), 256, 0, s>>>(perm, P.n_packed, (const uint64_t*)natural,
                                                             (uint64_t*)packed);
  else
    k_pack<uint32_t><<<blocks_for(P.n_packed), 256, 0, s>>>(perm, P.n_packed, (const uint32_t*)natural,
                                                             (uint32_t*)packed);
  return cudaGetLastError();
}

cudaError_t launch_unpack(const DevPlan& P, int elem_bytes, const void* packed, void* natural, cudaStream_t s) {
  if (P.n_packed == 0) return cudaSuccess;
  return elem_bytes == 8 ? unpack<uint64_t>(P, packed, natural, s) : unpack<uint32_t>(P, packed, natural, s);
}

}  // namespace hines
