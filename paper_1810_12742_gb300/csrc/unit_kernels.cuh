// Warp-task kernels of the batched Hines solver, sm_103a.
//
// The planner cuts every cell into units -- whole small cells, or the top part
// and the subtrees of a large cell -- and packs units into tasks.  A runner --
// a team of two warps, or a lone warp where teams would take more rounds of
// tasks (launch_phases) -- owns a task and walks its chunks (Hu's list schedule of the task's pieces, at most
// 32 * P pieces each, longest first): deepest chunk first for the
// elimination, root-side chunk first for the substitution (Section 3).  In a
// team one warp computes; the other moves data, so that copying a chunk's
// results out and staging the next chunk's inputs overlap the arithmetic
// (run_task).  Lane j of the computing warp owns the chunk's pieces P j ..
// P j + P - 1 (P = 1 or 2 pieces per lane).
// Inside a piece the parent of compartment i is i - 1 (Section 5): the lane
// runs a Thomas chain (Listing 1) and leaves one contribution for its parent
// compartment (Listing 2's parent lookup).  With P = 2 the lane runs its two
// chains at once, the two pieces aligned at their proximal ends (the shorter
// one joins the chain when its distal row comes up), so that both halves of
// every value live in one 8-byte register pair and the compensated
// arithmetic runs on packed FP32-pair instructions.
//
// A solve is two launches: (A) whole-cell tasks (both sweeps), the
// elimination of subtree tasks and, taken over by the runner that finishes a
// cell's last subtree, that cell's top part (both sweeps); (C) the
// substitution of subtree tasks.  No runner ever waits for another.
//
// The chunks of a task follow one another in the same runner, so a chunk's
// children are usually in the chunk just before it (elimination) and its
// parents likewise (substitution): those values pass through a small shared
// memory cache; other values go through global memory.  A chunk's inputs are
// staged into shared memory in the row layout of Section 5 (row r: the
// compartments r rows from each pair's distal start, one word per piece), so
// that a lane reads its P values of a row as one word: gathered with cp.async
// from the natural layout, or, where they are one contiguous block (the
// solver layout, and the factor blocks the eliminations leave in block
// order), by bulk copies one lane issues (BulkStage).
#pragma once
#include <cuda_runtime.h>

#include <cstdint>
#include <type_traits>

#include "../../include/hines.h"
#include "device_common.cuh"
#include "kernels.h"
#include "plan.h"

namespace hines {
namespace {

using namespace dev;

constexpr int kL = kBranchCap;          // rows (compartments per piece), at most
static_assert(kWarpsPerCta == 2, "a team: one computing and one moving warp");
constexpr int kSmemPerSm = 228 * 1024;  // shared memory of an SM; 1 KB of it goes to each resident CTA
// CTAs (teams) of `bytes` of shared memory an SM holds, at most `most`
constexpr int teams_per_sm(int bytes, int most) {
  return kSmemPerSm / (bytes + 16 + 1024) < most ? kSmemPerSm / (bytes + 16 + 1024) : most;
}

template <int P>
struct Geo {
  static constexpr int kChunk = 32 * P;              // pieces per chunk
  static constexpr int kS = P == 2 ? 66 : 32;        // natural staging: words per row
  static constexpr int kSlots = kL * kS + 4;         // words per staged array (holds a padded solver-layout block)
};
// Natural-layout staging: the word of piece i's compartment in row r.  One
// piece per lane: rows of 32 words, the column XOR-swizzled by the row, so
// that the warp's staging copies (sixteen consecutive rows of one piece per
// half-warp) and the lanes' row reads are both free of bank conflicts.  Two
// pieces per lane: rows of 66 words (64 + 2), so that a lane's pair is one
// aligned 8-byte word and the staging copies spread over the banks.
template <int P>
__device__ __forceinline__ int nidx(int r, int i) {
  if constexpr (P == 2)
    return r * 66 + i;
  else
    return (r << 5) + (i ^ (r & 31));
}
template <int P>
struct VOf {
  using type = float;
};
template <>
struct VOf<2> {
  using type = F2;
};

// ---- per-lane metadata ------------------------------------------------------
struct Piece {
  long long first, pcomp;  // natural: proximal compartment, parent compartment; solver layout: the chunk's
                           // block offset, the parent's solver-layout index (-1 at a cell's root)
  int ppos, child0, child1, len, nchild, ccontig, xtask;
};
// A parent's solution fetched ahead: a double-float pair (compensated and
// refinement modes) or one value of the solve's type (factor modes).
union PreX {
  float2 ff;
  float f;
  double d;
};
__device__ __forceinline__ float pre_get(const PreX& v, float) { return v.f; }
__device__ __forceinline__ double pre_get(const PreX& v, double) { return v.d; }
__device__ __forceinline__ void pre_set(PreX& v, float x) { v.f = x; }
__device__ __forceinline__ void pre_set(PreX& v, double x) { v.d = x; }

template <int P>
struct Meta {
  long long blk;  // the chunk's block offset in the solver layout
  Piece p[P];
  // substitution: the parent's solution when another chunk than the cached
  // predecessor left it, fetched a chunk ahead (fetch) so that its latency
  // overlaps the computation
  PreX xpre[P];
  // elimination (factor modes): the contributions of the first two children,
  // where other chunks than the cached predecessor left them, fetched likewise
  double2 cpre[P][2];
  int L;         // rows of the lane: length of its first (longer) piece, 0 for a lane without pieces
};

// The same as it lies in memory.  A chunk's records are loaded two chunks
// ahead and unpacked only when they are first needed: taking the packed fields
// apart right after the load waited for it in every chunk (about 600 clocks
// with one warp on the multiprocessor, 2000 to 2500 with all of them resident).
// With the chunk table in registers, the first entries without an atomic and
// the counters restored by the kernels instead of a copy: FP64 solve of 64
// small cells 52.7 -> 47.1 us, of 37 large cells 583 -> 554 us, FP32 solve of
// 1001 small cells 91.9 -> 81.0 us, compensated solve of 28M compartments
// 857 -> 835 us.
template <bool kPk, int P>
struct RawMeta {
  uint4 a[P], b[P];           // BrMetaT
  longlong2 pk[kPk ? P : 1];  // solver-layout record
  long long blk;
};
static_assert(sizeof(BrMetaT) == 32, "two 16-byte words");

template <bool kPk, int P>
__device__ __forceinline__ RawMeta<kPk, P> load_meta(const DevPlan& Pl, int c0, int n, int lane, bool want_blk) {
  RawMeta<kPk, P> m;
  m.blk = 0;
  if (want_blk && n > 0) m.blk = __ldg(&Pl.pk_meta[c0].x);  // every piece of a chunk shares it
#pragma unroll
  for (int h = 0; h < P; ++h) {
    const int i = P * lane + h;
    m.a[h] = make_uint4(0u, 0u, ~0u, ~0u);  // no piece: first 0, parents -1, length 0
    m.b[h] = make_uint4(~0u, 0u, 0u, 0u);  // (no children)
    if (kPk) m.pk[h] = make_longlong2(0, -1);
    if (i < n) {
      const uint4* t = reinterpret_cast<const uint4*>(Pl.tmeta + c0 + i);
      m.a[h] = __ldg(t);
      m.b[h] = __ldg(t + 1);
      if (kPk) m.pk[h] = __ldg(Pl.pk_meta + c0 + i);
    }
  }
  return m;
}

template <bool kPk, int P>
__device__ __forceinline__ Meta<P> unpack_meta(const RawMeta<kPk, P>& r) {
  Meta<P> m;
  m.blk = r.blk;
#pragma unroll
  for (int h = 0; h < P; ++h) {
    Piece& q = m.p[h];
    const uint4 a = r.a[h], b = r.b[h];
    q.first = kPk ? r.pk[h].x : (long long)(((unsigned long long)(a.y & 0xFFFFFFu) << 32) | a.x);
    q.pcomp = kPk ? r.pk[h].y : (long long)(((unsigned long long)a.w << 32) | a.z);
    q.ppos = (int)b.x;
    q.child0 = (int)b.y;
    q.child1 = (int)b.z;
    q.len = (int)(a.y >> 24);
    q.nchild = (int)(b.w & 0x3FFFFFFFu);
    q.ccontig = (int)((b.w >> 30) & 1u);
    q.xtask = (int)(b.w >> 31);
    m.xpre[h].d = 0.0;
    m.cpre[h][0] = m.cpre[h][1] = make_double2(0.0, 0.0);
  }
  m.L = m.p[0].len;
  return m;
}

// Position of child c: the first two children of a piece with at most two are
// in its record, so that their contributions need no dependent load.
__device__ __forceinline__ int child_pos(const DevPlan& Pl, const Piece& q, int c) {
  if (c == 0) return q.child0;
  if (q.nchild == 2) return q.child1;
  return q.ccontig ? q.child0 + c : __ldg(Pl.tchild + q.child1 + c);
}

// apply(load(c)) for the children of each lane's piece from child c on, in
// order.  In a lone warp's kernel (kAlone) the lanes of `live`, the callers,
// go in step, two children at a time: left to their own trip counts the lanes
// of the FP32 kernels stayed apart after the loop and ran the rows behind it in
// groups (FP32 solve of 1000 cells of 2000 compartments: 104 million warp
// instructions with 13 threads each, 392 us; in step 60 with 18, 198 us).  The
// teams' kernels do not, and lose 3 to 7% to the votes.
template <bool kAlone, typename Load, typename Apply>
__device__ __forceinline__ void for_children(unsigned live, int nchild, int c, Load&& load, Apply&& apply) {
  if constexpr (kAlone) {
#pragma unroll 1
    for (; __any_sync(live, c < nchild); c += 2) {
      if (c >= nchild) continue;
      const auto a = load(c);
      if (c + 1 < nchild) {
        const auto b = load(c + 1);
        apply(a);
        apply(b);
      } else {
        apply(a);
      }
    }
  } else {
#pragma unroll 1
    for (; c < nchild; ++c) apply(load(c));
  }
}

// A child's contribution slot: through L2 when another warp may have written
// it in this launch (a top part's subtree children), else the ordinary path.
template <typename W>
__device__ __forceinline__ W slot_load(const W* p, const Piece& q) {
  return q.xtask ? __ldcg(p) : *p;
}

// The chunk processed just before the current one in the same sweep.
struct Prev {
  int c0, n, which;  // n = 0: none
};

// ---- rows of the staged chunk -------------------------------------------------
// Word index of row r's first slot: natural layout, the fixed stride of the
// staging buffer; solver layout, the block's row offsets (a per-warp table).
template <bool kPk, int P>
struct Rows {
  const int* tab;
  // word of chunk position j (a lane's first piece: P * lane) in row r
  __device__ __forceinline__ int slot(int r, int j) const {
    if constexpr (kPk)
      return tab[r] + j;
    else
      return nidx<P>(r, j);
  }
};

// Solver layout: the row offsets of the current chunk's block from the lanes'
// row counts (every lane calls it); tab[kL] is the block's slot count.
template <int P>
__device__ __forceinline__ void build_row_table(int L, int lane, int* tab) {
  int acc = 0;
#pragma unroll
  for (int r = 0; r < kL; ++r) {
    const int nl = __popc(__ballot_sync(kFull, L > r));
    if (lane == r) tab[r] = acc;
    acc += P * nl;
  }
  if (lane == 0) tab[kL] = acc;
  __syncwarp();
}

// Piece i of the chunk (its owner lane's metadata, by shuffle; every lane calls it).
struct ChunkElem {
  long long first;
  int len, rows;  // compartments; rows of the owner lane
};
template <int P>
__device__ __forceinline__ ChunkElem chunk_elem(const Meta<P>& m, int i) {
  const int src = (i / P) & 31;
  // first (below 2^34) and length in one word
  auto packed = [&](int h) { return (unsigned long long)m.p[h].first | (unsigned long long)m.p[h].len << 40; };
  unsigned long long w = __shfl_sync(kFull, packed(0), src);
  int rows = 0;
  if constexpr (P == 2) {
    rows = __shfl_sync(kFull, m.L, src);
    const unsigned long long w1 = __shfl_sync(kFull, packed(1), src);
    if (i & 1) w = w1;
  }
  ChunkElem c{(long long)(w & ((1ull << 40) - 1)), (int)(w >> 40), rows};
  if constexpr (P == 1) c.rows = c.len;
  return c;
}

// Every element of the chunk's pieces in the natural layout: sixteen lanes
// per piece, two pieces per step (pieces are at most 16 long).  f(i, t, row,
// g) for piece i, distance t from its proximal end, row of the staged chunk,
// natural index g.
template <int P, typename F>
__device__ __forceinline__ void for_chunk_elements(const Meta<P>& m, int n, int lane, F&& f) {
  const int half = lane >> 4, t = lane & 15;
#pragma unroll 1
  for (int j = 0; j < n; j += 2) {
    const int i = j + half;
    const ChunkElem c = chunk_elem(m, i);
    if (i < n && t < c.len) f(i, t, c.rows - 1 - t, c.first + t);
  }
}

// Solver layout: copy the chunk's block of one array into shared memory with
// 16-byte copies (blocks start on multiples of 4 slots and are padded).
template <typename T>
__device__ __forceinline__ void stage_block(T* dst, const T* src, long long blk, int e, int lane) {
  constexpr int V = 16 / (int)sizeof(T);
  const int nv = (e + V - 1) / V;
#pragma unroll 1
  for (int v = lane; v < nv; v += 32) cp_async16(dst + v * V, src + blk + (long long)v * V);
}

// ---- one or two values of a row -------------------------------------------------
__device__ __forceinline__ float ldv(const float* s, int idx, float) { return s[idx]; }
__device__ __forceinline__ F2 ldv(const float* s, int idx, F2) { return *reinterpret_cast<const F2*>(s + idx); }
__device__ __forceinline__ void stv(float* s, int idx, float v) { s[idx] = v; }
__device__ __forceinline__ void stv(float* s, int idx, F2 v) { *reinterpret_cast<F2*>(s + idx) = v; }
__device__ __forceinline__ float vget(float v, int) { return v; }
__device__ __forceinline__ float vget(F2 v, int h) { return h == 0 ? f2_lo(v) : f2_hi(v); }
template <int P>
__device__ __forceinline__ typename VOf<P>::type vpack(const float* a) {
  if constexpr (P == 2)
    return f2_make(a[0], a[1]);
  else
    return a[0];
}
// the second half of v replaced by w (the shorter piece joins its chain)
__device__ __forceinline__ F2 vset_hi(F2 v, float w) { return f2_make(f2_lo(v), w); }

// ---- bulk staging -------------------------------------------------------------
// Contiguous blocks are staged by one-dimensional bulk copies that one lane of
// the moving warp issues, completing on the staging buffer's shared-memory
// barrier at its byte kOff (then its phase parity and a failure flag), on
// which the computing warp waits.
template <int kOff>
struct BulkStage {
  static_assert(kOff % 8 == 0, "barrier alignment");
  // bounded wait: a poll that sees nothing suspends about 3.75 us on a GB300
  // (hines_check_bounded_wait measures it), so about one second in all, far
  // beyond any real copy latency
  static constexpr int kWaitPolls = 1 << 18;
  __device__ static uint64_t* barrier(unsigned char* buf) { return reinterpret_cast<uint64_t*>(buf + kOff); }
  __device__ static unsigned* words(unsigned char* buf) { return reinterpret_cast<unsigned*>(barrier(buf) + 1); }
  // once per staging buffer, before the first task (one thread)
  __device__ static void init(unsigned char* buf) {
    mbar_init(barrier(buf));
    words(buf)[0] = 0u;  // parity of the next phase
    words(buf)[1] = 0u;  // a wait on this buffer has run out
  }
  // one arrival with the expected bytes, then the copies.  Every lane fences
  // its earlier ordinary accesses to the buffer first (the computing warp's
  // lie before the team's last barrier); what the copies read of this task's
  // own results is fenced where the sweeps turn (run_task).
  template <int N>
  __device__ static void issue(unsigned char* buf, int lane, unsigned bytes, void* d0, const void* s0,
                               void* d1 = nullptr, const void* s1 = nullptr, void* d2 = nullptr,
                               const void* s2 = nullptr) {
    fence_async_shared();
    __syncwarp();
    if (lane == 0) {
      uint64_t* bar = barrier(buf);
      mbar_expect_tx(bar, N * bytes);
      if (bytes > 0) {
        bulk_g2s(d0, s0, bytes, bar);
        if (N > 1) bulk_g2s(d1, s1, bytes, bar);
        if (N > 2) bulk_g2s(d2, s2, bytes, bar);
      }
    }
  }
  // every lane waits for the staged copies; a wait that runs out raises the
  // plan's timeout status and goes on (no access leaves its buffer), and
  // later waits on the buffer poll only once, so that a failed launch ends within
  // about a second instead of a second per chunk
  __device__ static void wait(const DevPlan& Pl, unsigned char* buf, int lane) {
    unsigned* w = words(buf);
    const unsigned parity = w[0];
    const bool ok = mbar_wait(barrier(buf), parity, w[1] ? 1 : kWaitPolls);
    if (!ok && lane == 0 && Pl.status) atomicCAS(Pl.status, 0, (int)HINES_ERR_TIMEOUT);
    __syncwarp();
    if (lane == 0) {
      w[0] = parity ^ 1u;
      if (!ok) w[1] = 1u;
    }
    __syncwarp();
  }
};

// ============================================================================
// Compensated mode: FP32 inputs, double-float arithmetic from FP32 error-free
// transformations, FP64 solution.  The elimination leaves, per compartment k,
// the two double-float numbers the substitution needs, y_k = B_k / D_k and
// g_k = u_k / D_k (D, B: the eliminated pivot and right-hand side), written
// in the chunk's block order of the solver layout (16 bytes a slot, each row
// a contiguous run); per piece its contribution to the parent.  The
// substitution stages the block with 16-byte copies and runs
// x_k = y_k - g_k x_{k+1} from the proximal row (x of the parent's distal
// compartment) to the distal one: no inputs are read again.
// ============================================================================
template <bool kPk, int P>
struct CompMode {
  using V = typename VOf<P>::type;
  using G = Geo<P>;
  static constexpr bool kPacked = kPk;
  static constexpr bool kNeedsBlk = true;
  static constexpr int kPer = P;
  // row loops: the natural layout's longer chunk code does better in fewer
  // copies (28M compartments 833 against 891 us), the solver layout's does not
  // (21M with the unpack 836 against 827 us)
  static constexpr int kUnroll = kPk ? kL : 4;
  struct Args {
    const float* d;
    const float* u;
    const float* b;
    double* x;
  };
  // a staging buffer: elimination, d, u, b (3 words a slot); substitution,
  // the factor block (4 words a slot, the FP64 solution written over its
  // first two); then the block's row table
  static constexpr int kArr = 3 * G::kSlots * 4, kFac = G::kSlots * 16;
  static constexpr int kTab = kArr > kFac ? kArr : kFac;
  static constexpr int kStageBytes = kTab + 96;
  // the caches of the two sweeps share their space
  static constexpr int kCslot = 0, kCx = 0, kCacheBytes = 2 * G::kChunk * 16;
  static constexpr int kTeamBytes = 2 * kStageBytes + kCacheBytes;
  static constexpr int kWarpBytes = kStageBytes + kCacheBytes;
  static constexpr int kMinBlocks = teams_per_sm(kTeamBytes, 12), kMinBlocksAlone = teams_per_sm(2 * kWarpBytes, 12);
  // teams in phase A up to this many sixteenths of an entry per resident team
  // (team against lone warp, us a solve: 1940 entries 240 : 290, 1421 377 :
  // 414; phase A alone, 2370 entries 535 : 573; solver layout, whose copies are
  // bulk copies, 1197 381 : 412, 2629 665 : 601)
  static constexpr int kTeamShare = kPk ? 18 : 24;
  // a team's speed at a chunk against a lone warp's (one task each: 1.15 to
  // 1.26, solver layout 1.0 to 1.06)
  static constexpr double kTeamSpeed = kPk ? 1.15 : 1.25;
  static_assert(kStageBytes % 16 == 0, "16-byte aligned buffers");
  // contiguous blocks (the factor block; d, u, b in the solver layout) are
  // staged by bulk copies, the barrier after the row table
  using Bulk = BulkStage<kTab + 80>;

  __device__ static bool bulk_staged(int visit) { return visit == 1 || kPk; }
  __device__ static void init_buffer(unsigned char* buf) { Bulk::init(buf); }
  // what the chunk needs of earlier chunks that no cache holds
  template <bool kAlone>
  __device__ static void fetch(const DevPlan& Pl, const Args&, int visit, Meta<P>& m, const Prev& pv) {
    if (visit == 0) return;
#pragma unroll
    for (int h = 0; h < P; ++h) {
      const Piece& q = m.p[h];
      const int loc = q.ppos - pv.c0;
      if (q.len > 0 && q.pcomp >= 0 && !(loc >= 0 && loc < pv.n))
        m.xpre[h].ff = static_cast<const float2*>(Pl.xlast)[q.ppos];
    }
  }

  __device__ static void stage(const DevPlan& Pl, const Args& A, int visit, const Meta<P>& m, int n, int lane,
                               unsigned char* buf) {
    int* tab = reinterpret_cast<int*>(buf + kTab);
    build_row_table<P>(m.L, lane, tab);
    const int e = tab[kL];
    if (visit == 1) {
      Bulk::template issue<1>(buf, lane, (unsigned)e * 16u, buf, static_cast<const float4*>(Pl.ff4) + m.blk);
      return;
    }
    float* sd = reinterpret_cast<float*>(buf);
    float* su = sd + G::kSlots;
    float* sb = su + G::kSlots;
    if (kPk) {
      const long long blk = __shfl_sync(kFull, m.p[0].first, 0);
      // whole 16-byte words: the block's padding (blocks start on multiples
      // of 4 slots, and the layout's length is one) completes the last
      Bulk::template issue<3>(buf, lane, (unsigned)((e + 3) & ~3) * 4u, sd, A.d + blk, su, A.u + blk, sb, A.b + blk);
      return;
    }
    for_chunk_elements(m, n, lane, [&](int i, int, int row, long long g) {
      const int q = nidx<P>(row, i);
      cp_async4(&sd[q], A.d + g);
      cp_async4(&su[q], A.u + g);
      cp_async4(&sb[q], A.b + g);
    });
    cp_commit();
  }

  template <bool kAlone>
  __device__ static void compute(const DevPlan& Pl, const Args&, int visit, int c0, int n, int lane,
                                 const Meta<P>& m, unsigned char* buf, const Prev& pv, unsigned char* cache, int cur) {
    float4* cslot = reinterpret_cast<float4*>(cache + kCslot);  // [2][kChunk] contributions
    float2* cx = reinterpret_cast<float2*>(cache + kCx);        // [2][kChunk] distal solutions
    const int* tab = reinterpret_cast<const int*>(buf + kTab);
    float4* slot = static_cast<float4*>(Pl.cd);
    float2* xlast = static_cast<float2*>(Pl.xlast);
    if (bulk_staged(visit)) Bulk::wait(Pl, buf, lane);
    const int L = m.L;
    const unsigned live = kAlone ? __ballot_sync(kFull, L > 0) : 0u;  // (for_children)
    if (L == 0) return;
    const int me = P * lane;
    // the second piece's distal row (it joins the chain there); L: none
    const int delta = P == 2 ? L - m.p[P - 1].len : 0;
    if (visit == 0) {
      const float* sd = reinterpret_cast<const float*>(buf);
      const float* su = sd + G::kSlots;
      const float* sb = su + G::kSlots;
      float4* fac = static_cast<float4*>(Pl.ff4) + m.blk;
      const Rows<kPk, P> rows{tab};
      float d0h[P], d0l[P], b0h[P], b0l[P];
#pragma unroll
      for (int h = 0; h < P; ++h) {
        const Piece& q = m.p[h];
        d0h[h] = 1.f;
        d0l[h] = b0h[h] = b0l[h] = 0.f;
        if (!kAlone && q.len == 0) continue;  // (a lone warp's lanes go on together)
        const int idx = q.len > 0 ? rows.slot(L - q.len, me + h) : 0;
        ff Dv = {q.len > 0 ? sd[idx] : 1.f, 0.f}, Bv = {q.len > 0 ? sb[idx] : 0.f, 0.f};
        for_children<kAlone>(
            live, q.nchild, 0,
            [&](int c) {
              const int cp = child_pos(Pl, q, c);
              const int loc = cp - pv.c0;
              return (loc >= 0 && loc < pv.n) ? cslot[pv.which * G::kChunk + loc] : slot_load(slot + cp, q);
            },
            [&](const float4& v) {
              Dv = ff_sub(Dv, v.x, v.y);
              Bv = ff_sub(Bv, v.z, v.w);
            });
        d0h[h] = Dv.h;
        d0l[h] = Dv.l;
        b0h[h] = Bv.h;
        b0l[h] = Bv.l;
      }
      FFV<V> D{vpack<P>(d0h), vpack<P>(d0l)}, B{vpack<P>(b0h), vpack<P>(b0l)};
      // row r: g = u / D, y = B / D into the factor block; then the chain to row r + 1
#pragma unroll kUnroll
      for (int r = 0; r < kL - 1; ++r) {
        if (r < L - 1) {
          const V uk = ldv(su, rows.slot(r, me), V{});
          const FFV<V> g = vdiv_f(uk, D);
          const FFV<V> y = vdiv(B, D);
          const int f0 = tab[r] + me;
#pragma unroll
          for (int h = 0; h < P; ++h)
            fac[f0 + h] = make_float4(vget(y.h, h), vget(y.l, h), vget(g.h, h), vget(g.l, h));
          const FFV<V> fu = vmul_f(g, uk);
          const FFV<V> fb = vmul_ff(g, B);
          const int i1 = rows.slot(r + 1, me);
          D = vsub_dom(ldv(sd, i1, V{}), fu.h, fu.l);
          B = vsub_ff(ldv(sb, i1, V{}), fb.h, fb.l);
          if constexpr (P == 2) {
            if (r + 1 == delta) {
              D = {vset_hi(D.h, d0h[1]), vset_hi(D.l, d0l[1])};
              B = {vset_hi(B.h, b0h[1]), vset_hi(B.l, b0l[1])};
            }
          }
        }
      }
      // the proximal row: its factor, and the contribution to the parent (a
      // root's solution is its y, the factor's first number)
      const V uk = ldv(su, rows.slot(L - 1, me), V{});
      const FFV<V> g = vdiv_f(uk, D);
      const FFV<V> y = vdiv(B, D);
      const FFV<V> fu = vmul_f(g, uk);
      const FFV<V> fb = vmul_ff(g, B);
      const int f0 = tab[L - 1] + me;
#pragma unroll
      for (int h = 0; h < P; ++h) {
        const bool root = m.p[h].pcomp < 0;  // a cell's root: no coupling to a parent
        fac[f0 + h] = make_float4(vget(y.h, h), vget(y.l, h), root ? 0.f : vget(g.h, h), root ? 0.f : vget(g.l, h));
        if (m.p[h].len == 0 || root) continue;
        const float4 out = make_float4(vget(fu.h, h), vget(fu.l, h), vget(fb.h, h), vget(fb.l, h));
        slot[c0 + me + h] = out;
        cslot[cur * G::kChunk + me + h] = out;
      }
      return;
    }
    // substitution: x = y - g x_parent from the proximal row down; the FP64
    // solution goes over the slot's first two words
    float4* sf = reinterpret_cast<float4*>(buf);
    float xph[P], xpl[P];
#pragma unroll
    for (int h = 0; h < P; ++h) {
      const Piece& q = m.p[h];
      xph[h] = xpl[h] = 0.f;
      if (q.len > 0 && q.pcomp >= 0) {
        const int loc = q.ppos - pv.c0;
        const float2 t = (loc >= 0 && loc < pv.n) ? cx[pv.which * G::kChunk + loc] : m.xpre[h].ff;
        xph[h] = t.x;
        xpl[h] = t.y;
      }
    }
    FFV<V> X{vpack<P>(xph), vpack<P>(xpl)};
    float xbh = 0.f, xbl = 0.f;  // the second piece's distal solution
    // a row's factor is read before the row above it writes its solution (the
    // compiler may not move the read over the write)
    float4 f[P];
#pragma unroll
    for (int h = 0; h < P; ++h) f[h] = sf[tab[L - 1] + me + h];
#pragma unroll kUnroll
    for (int r = kL - 1; r >= 0; --r) {
      if (r < L) {
        const int q = tab[r] + me;
        float yh[P], yl[P], gh[P], gl[P];
#pragma unroll
        for (int h = 0; h < P; ++h) {
          yh[h] = f[h].x;
          yl[h] = f[h].y;
          gh[h] = f[h].z;
          gl[h] = f[h].w;
          if (r > 0) f[h] = sf[tab[r - 1] + me + h];
        }
        const FFV<V> gx = vmul_ff(FFV<V>{vpack<P>(gh), vpack<P>(gl)}, X);
        X = vsub_ffff(FFV<V>{vpack<P>(yh), vpack<P>(yl)}, gx.h, gx.l);
#pragma unroll
        for (int h = 0; h < P; ++h)
          reinterpret_cast<double*>(sf + q + h)[0] = ff_to_double(vget(X.h, h), vget(X.l, h));
        if constexpr (P == 2) {
          if (r == delta) {
            xbh = f2_hi(X.h);
            xbl = f2_hi(X.l);
          }
        }
      }
    }
#pragma unroll
    for (int h = 0; h < P; ++h) {
      if (m.p[h].len == 0) continue;
      const float2 xo = h == 0 ? make_float2(vget(X.h, 0), vget(X.l, 0)) : make_float2(xbh, xbl);
      xlast[c0 + me + h] = xo;
      cx[cur * G::kChunk + me + h] = xo;
    }
  }

  __device__ static void copy_out(const DevPlan&, const Args& A, int visit, const Meta<P>& m, int n, int lane,
                                  unsigned char* buf) {
    if (visit == 0) return;
    const double* sx = reinterpret_cast<const double*>(buf);  // two per slot: the solution, then g
    const int* tab = reinterpret_cast<const int*>(buf + kTab);
    if (kPk) {
      const long long blk = __shfl_sync(kFull, m.p[0].first, 0);
      const int e = tab[kL];
#pragma unroll 1
      for (int s = lane; s < e; s += 32) A.x[blk + s] = sx[2 * s];
      return;
    }
    for_chunk_elements(m, n, lane, [&](int i, int, int row, long long g) { A.x[g] = sx[2 * (tab[row] + i)]; });
  }
};

// ============================================================================
// Factor mode (FP64, FP32, passive cable).  FP64: the elimination leaves, per
// compartment, g = u / D and y = B / D (D, B: the eliminated pivot and
// right-hand side), and the substitution runs x = y - g x_parent: one FP64
// instruction a row, no input read again.  The pair goes either into the
// plan's factor block, 16 bytes in the chunk's block order of the solver
// layout (each row a contiguous run), staged back with bulk copies, or to
// natural (or slot) positions, g into the workspace and y in place.  A full
// cable step or cable solve also leaves the reciprocal pivot, which steps that
// re-use the factor need for y.  FP32: the reciprocal pivot goes to the workspace and the
// right-hand side in place (the refinement reads that factor); the
// substitution reads them and u back.  In cable mode
// the system is rebuilt while staging (Section 1's implicit-Euler system):
// d_i = s_i (1 + theta dt g_i) + sum of a over the edges at i (a = -u),
// b_i = s_i V_i + s_i dt g_i (E - (1 - theta) V_i).
// The lane's pieces are handled one after the other in the same loop step
// (no packed FP64 instructions exist), their rows aligned as in the compensated
// mode; a piece's rows before its distal row are skipped.
//
// The cable matrix is eliminated without its subtractions: with
// E_i = s_i (1 + theta dt g_i) + sum over the children c of a_c E_c / D_c, the
// conductance to ground seen at i, the pivot is D_i = E_i + a_i (a cell's
// root: E_i), since a_c - a_c^2 / D_c = a_c E_c / D_c.  The same number of
// operations, and nothing cancels where the leak is small next to a.
//
// The FP64 pipe and the latency of a row bound this mode: an FP64 instruction
// takes a scheduler 64 to 76 clocks (64 of latency), so a row holds as few of
// them as possible (elimination 4, cable 5, substitution 1), and the
// next row's inputs are read before the current row's results are written
// (the compiler may not move them over the stores).
// ============================================================================
// kReuse: a passive-cable step with the factor a full step of the same plan
// and matrix left in the workspace: only the right-hand side is rebuilt and
// eliminated.
// kBlk: FP64 keeps its factor in block order (else at natural positions, as
// FP32 always does).
template <typename T, bool kCable, bool kPk, int P, bool kReuse = false, bool kBlk = true>
struct FactorMode {
  using G = Geo<P>;
  // the reciprocal eliminated diagonal: FP64 as rcp_t gives it; FP32 with one
  // more Newton step on the hardware approximation, so that the stored factor
  // is that of an FP32 elimination to the last bit or so, which the
  // refinement's re-solves depend on
  __device__ static T rcp_solve(T x) {
    T r = rcp_t(x);
    if (sizeof(T) == 4) r = fma(r, fma(-x, r, T(1)), r);
    return r;
  }
  static constexpr bool kPacked = kPk;
  static constexpr bool kYG = sizeof(T) == 8;  // the factor is (g, y)
  static constexpr bool kBF = kBlk && kYG;     // ... in block order
  static constexpr bool kNeedsBlk = kBF;
  static constexpr int kPer = P;
  // row loops: sixteen copies of the long FP64 row overrun the instruction
  // cache (2 against 16: 64 small cells 47.1 against 51.2 us, 59M compartments
  // 1.61 against 1.65 ms); a row that re-uses its factor is short (7.85
  // against 7.29 ms per 40 steps of 1.7M compartments)
  static constexpr int kUnroll = kYG && !kReuse ? 2 : kL;
  static_assert(!kReuse || (kCable && kYG), "only FP64 cable steps re-use a factor");
  struct Args {
    const T* d;
    const T* u;
    const T* s;  // cable: s, g
    const T* g;
    T* x;        // right-hand side in, solution out (cable: V in, V out)
    T dt, E, theta;
    bool rhs_from_V;  // cable: a time step (else a solve with the step's matrix)
    const T* rhs = nullptr;  // non-null: the right-hand side is read from here (x receives the solution)
  };
  // a staging buffer: d (or the factor), u, b, then the row table (solver layout)
  static constexpr int kTab = 3 * G::kSlots * (int)sizeof(T);
  static constexpr int kStageBytes = kTab + 96;
  static constexpr int kCslot = 0, kCx = 0, kCacheBytes = 2 * G::kChunk * 2 * (int)sizeof(T);
  static constexpr int kTeamBytes = 2 * kStageBytes + kCacheBytes;
  static constexpr int kWarpBytes = kStageBytes + kCacheBytes;
  static constexpr int kMinBlocks = teams_per_sm(kTeamBytes, 10), kMinBlocksAlone = teams_per_sm(2 * kWarpBytes, 10);
  // the same (us; FP64: 1440 entries 262 : 318, 1514 668 : 764, 2184 376 :
  // 392, 2260 586 : 628, 2707 542 : 509, 2755 954 : 953; FP32: 1514 162 : 205,
  // 2370 592 : 639, 2618 380 : 399; re-using a factor: 2184 2511 : 2817, 2700
  // 5731 : 5727)
  static constexpr int kTeamShare = kReuse ? 40 : 32;
  // one task each: FP64 and FP32 1.15 to 1.29, cable 1.18 to 1.23, re-using a
  // factor 1.32; stretch 1.31 (1024 uneven cells): FP64 929 : 977, cable step
  // 1514 : 1371
  static constexpr double kTeamSpeed = kCable && !kReuse ? 1.25 : sizeof(T) == 4 ? 1.3 : 1.35;
  // the factor block is staged by bulk copies
  static constexpr bool kBulk = kBF;
  static_assert(kStageBytes % 16 == 0, "16-byte aligned buffers");
  using Bulk = BulkStage<kTab + 80>;
  __device__ static void init_buffer(unsigned char* buf) {
    if (kBulk) Bulk::init(buf);
  }
  // (g, y) per slot of the solver layout
  __device__ static double2* factor_block(const DevPlan& Pl) { return static_cast<double2*>(Pl.ff4); }
  // the reciprocal pivots of the last full elimination: the workspace the other placement's factor would use
  __device__ static T* reciprocals(const DevPlan& Pl) { return static_cast<T*>(kBF ? Pl.fac : Pl.ff4); }
  __device__ static bool keeps_rcp(const Args&) { return kYG && kCable && !kReuse; }

  // Section 1's implicit-Euler system, each part in the fewest operations: the
  // diagonal less all its edges, s (1 + theta dt g), and the right-hand side
  // s (V + dt g (E - (1 - theta) V)) (theta = 1: s (V + dt E g))
  __device__ static T cable_diag(const Args& A, T si, T gi) { return si * fma(A.theta * A.dt, gi, T(1)); }
  __device__ static T cable_rhs(const Args& A, T si, T gi, T vi) {
    if (A.theta == T(1)) return si * fma(A.dt * A.E, gi, vi);
    return si * fma(A.dt * gi, fma(A.theta - T(1), vi, A.E), vi);
  }

  // Rebuild of the chunk's system (cable, elimination).  kStep elements per
  // lane are loaded before any is computed: one at a time, every element
  // waited for its loads (19.6k clocks a chunk of the 15M-compartment step,
  // more than the elimination itself).
  static constexpr int kStep = 2;
  struct Elem {
    T s, g, u, v;
    __device__ void load(const Args& A, long long i) {
      v = A.x[i];
      if (!kReuse) u = A.u[i];
      if (!kReuse || A.rhs_from_V) {
        s = A.s[i];
        g = A.g[i];
      }
    }
    __device__ void store(const Args& A, T* sd, T* su, T* sb, int q) const {
      if (!kReuse) {
        sd[q] = cable_diag(A, s, g);
        su[q] = u;
      }
      sb[q] = A.rhs_from_V ? cable_rhs(A, s, g, v) : v;
    }
  };
  __device__ static void rebuild_block(const Args& A, long long blk, int e, int lane, T* sd, T* su, T* sb) {
#pragma unroll 1
    for (int i0 = lane; i0 < e; i0 += 32 * kStep) {
      Elem el[kStep];
#pragma unroll
      for (int k = 0; k < kStep; ++k)
        if (i0 + 32 * k < e) el[k].load(A, blk + i0 + 32 * k);
#pragma unroll
      for (int k = 0; k < kStep; ++k)
        if (i0 + 32 * k < e) el[k].store(A, sd, su, sb, i0 + 32 * k);
    }
  }
  template <typename F>
  __device__ static void rebuild_natural(const Args& A, const Meta<P>& m, int n, int lane, T* sd, T* su, T* sb, F&& f) {
    const int half = lane >> 4, t = lane & 15;
#pragma unroll 1
    for (int j = 0; j < n; j += 2 * kStep) {
      Elem el[kStep];
      int q[kStep];  // word of the staged chunk, -1: none
#pragma unroll
      for (int k = 0; k < kStep; ++k) {
        const int i = j + 2 * k + half;
        const ChunkElem c = chunk_elem(m, i);
        q[k] = i < n && t < c.len ? nidx<P>(c.rows - 1 - t, i) : -1;
        if (q[k] >= 0) {
          el[k].load(A, c.first + t);
          f(i, c.rows - 1 - t, q[k], c.first + t);
        }
      }
#pragma unroll
      for (int k = 0; k < kStep; ++k)
        if (q[k] >= 0) el[k].store(A, sd, su, sb, q[k]);
    }
  }

  // A child's contribution (D, B): from the cache of the chunk just before,
  // or from the slots.
  __device__ static bool local_child(int cp, const Prev& pv) { return cp >= pv.c0 && cp < pv.c0 + pv.n; }
  // what the chunk needs of earlier chunks that no cache holds: a parent's
  // solution, the contributions of the first two children (FP32: in lone
  // warps, whose solver-layout kernel takes 148 us with it and 260 without on
  // 1000 cells of 2000 compartments; teams gain nothing)
  template <bool kAlone>
  __device__ static constexpr bool fetches_children() {
    return kYG || kAlone;
  }
  template <bool kAlone>
  __device__ static void fetch(const DevPlan& Pl, const Args&, int visit, Meta<P>& m, const Prev& pv) {
#pragma unroll
    for (int h = 0; h < P; ++h) {
      const Piece& q = m.p[h];
      if (visit == 1) {
        const int loc = q.ppos - pv.c0;
        if (q.len > 0 && q.pcomp >= 0 && !(loc >= 0 && loc < pv.n))
          pre_set(m.xpre[h], static_cast<const T*>(Pl.xlast)[q.ppos]);
      } else if (fetches_children<kAlone>()) {
        using T2 = std::conditional_t<kYG, double2, float2>;
        const T2* slot = static_cast<const T2*>(Pl.cd);
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          if (c >= q.nchild) continue;
          const int cp = child_pos(Pl, q, c);
          if (local_child(cp, pv)) continue;
          const T2 v = slot_load(slot + cp, q);
          m.cpre[h][c] = make_double2(v.x, v.y);
        }
      }
    }
  }

  __device__ static void stage(const DevPlan& Pl, const Args& A, int visit, const Meta<P>& m, int n, int lane,
                               unsigned char* buf) {
    T* sd = reinterpret_cast<T*>(buf);
    T* su = sd + G::kSlots;
    T* sb = su + G::kSlots;
    int* tab = reinterpret_cast<int*>(buf + kTab);
    T* fac = static_cast<T*>(Pl.fac);
    if (kBF || kPk) build_row_table<P>(m.L, lane, tab);
    const int e = (kBF || kPk) ? tab[kL] : 0;
    const long long blk = kPk ? __shfl_sync(kFull, m.p[0].first, 0) : 0;
    if (visit == 1) {
      if constexpr (kBF) {  // the factor block over the first two arrays
        Bulk::template issue<1>(buf, lane, (unsigned)e * 16u, buf, factor_block(Pl) + m.blk);
      } else if (kPk) {
        stage_block(sd, static_cast<const T*>(fac), blk, e, lane);
        if (!kYG) stage_block(su, A.u, blk, e, lane);
        stage_block(sb, static_cast<const T*>(A.x), blk, e, lane);
        cp_commit();
      } else {
        for_chunk_elements(m, n, lane, [&](int i, int, int row, long long g) {
          const int q = nidx<P>(row, i);
          cp_async(&sd[q], fac + g);
          if (!kYG) cp_async(&su[q], A.u + g);
          cp_async(&sb[q], static_cast<const T*>(A.x) + g);
        });
        cp_commit();
      }
      return;
    }
    if constexpr (kReuse) {
      // the stored reciprocals and g, and the right-hand side rebuilt
      const T* rc = reciprocals(Pl);
      const T* gp = kBF ? reinterpret_cast<const T*>(factor_block(Pl) + m.blk) : fac;  // g: every other word, or by index
      if (kPk) {
        stage_block(sd, rc, blk, e, lane);
        if (kBF)
#pragma unroll 1
          for (int i = lane; i < e; i += 32) cp_async(&su[i], gp + 2 * i);
        else
          stage_block(su, gp, blk, e, lane);
        rebuild_block(A, blk, e, lane, sd, su, sb);
      } else {
        rebuild_natural(A, m, n, lane, sd, su, sb, [&](int i, int row, int q, long long g) {
          cp_async(&sd[q], kBF ? rc + m.blk + tab[row] + i : rc + g);
          cp_async(&su[q], kBF ? gp + 2 * (tab[row] + i) : gp + g);
        });
      }
    } else if constexpr (kCable) {
      if (kPk)
        rebuild_block(A, blk, e, lane, sd, su, sb);
      else
        rebuild_natural(A, m, n, lane, sd, su, sb, [](int, int, int, long long) {});
    } else {
      const T* bsrc = A.rhs ? A.rhs : static_cast<const T*>(A.x);
      if (kPk) {
        stage_block(sd, A.d, blk, e, lane);
        stage_block(su, A.u, blk, e, lane);
        stage_block(sb, bsrc, blk, e, lane);
      } else {
        for_chunk_elements(m, n, lane, [&](int i, int, int row, long long g) {
          const int q = nidx<P>(row, i);
          cp_async(&sd[q], A.d + g);
          cp_async(&su[q], A.u + g);
          cp_async(&sb[q], bsrc + g);
        });
      }
    }
    cp_commit();
  }

  template <bool kAlone>
  __device__ static void compute(const DevPlan& Pl, const Args& A, int visit, int c0, int n, int lane,
                                 const Meta<P>& m, unsigned char* buf, const Prev& pv, unsigned char* cache, int cur) {
    T* sd = reinterpret_cast<T*>(buf);
    T* su = sd + G::kSlots;
    T* sb = su + G::kSlots;
    T* cslot = reinterpret_cast<T*>(cache + kCslot);  // [2][kChunk][2] contributions
    T* cx = reinterpret_cast<T*>(cache + kCx);        // [2][kChunk] distal solutions
    T* slot = static_cast<T*>(Pl.cd);                 // [nb][2]
    const int* tab = reinterpret_cast<const int*>(buf + kTab);
    const Rows<kPk, P> rows{tab};
    if (kBulk && visit == 1) Bulk::wait(Pl, buf, lane);
    const int L = m.L;
    const unsigned live = kAlone ? __ballot_sync(kFull, L > 0) : 0u;  // (for_children)
    if (L == 0) return;
    const int me = P * lane;
    double2* bf = kBF ? factor_block(Pl) + m.blk : nullptr;  // the chunk's factor block
    int first_row[P];  // each piece's distal row
#pragma unroll
    for (int h = 0; h < P; ++h) first_row[h] = m.p[h].len > 0 ? L - m.p[h].len : kL;
    if (visit == 0) {
      const bool keep_rcp = keeps_rcp(A);
      T* rcp_block = kBF ? reciprocals(Pl) + m.blk : nullptr;
      // per piece: the eliminated pivot (cable: E) and right-hand side of the
      // current row, its coupling (re-using a factor: its g) and stored
      // reciprocal
      T D[P], B[P], uk[P], rk[P];
#pragma unroll
      for (int h = 0; h < P; ++h) {
        const Piece& q = m.p[h];
        D[h] = T(1);
        B[h] = uk[h] = rk[h] = T(0);
        if (!kAlone && q.len == 0) continue;  // (a lone warp's lanes go on together)
        if (q.len > 0) {
          const int idx = rows.slot(first_row[h], me + h);
          (kReuse ? rk[h] : D[h]) = sd[idx];
          B[h] = sb[idx];
          uk[h] = su[idx];
        }
        struct Contribution {
          T cd, cb;
        };
        auto load = [&](int c, double2 pre, bool fetched) {
          const int cp = child_pos(Pl, q, c);
          const int w = (pv.which * G::kChunk + cp - pv.c0) * 2;
          Contribution v;
          if (local_child(cp, pv)) {
            v.cd = kReuse ? T(0) : cslot[w];
            v.cb = cslot[w + 1];
          } else if (fetched) {
            v.cd = (T)pre.x;
            v.cb = (T)pre.y;
          } else {
            v.cd = kReuse ? T(0) : slot_load(slot + 2 * (size_t)cp, q);
            v.cb = slot_load(slot + 2 * (size_t)cp + 1, q);
          }
          return v;
        };
        auto apply = [&](const Contribution& v) {
          if (!kReuse) D[h] -= v.cd;
          B[h] -= v.cb;
        };
        constexpr bool kPre = fetches_children<kAlone>();
        if (kPre) {
          if (q.nchild > 0) apply(load(0, m.cpre[h][0], true));
          if (q.nchild > 1) apply(load(1, m.cpre[h][1], true));
        }
        for_children<kAlone>(
            live, q.nchild, kPre ? 2 : 0, [&](int c) { return load(c, make_double2(0.0, 0.0), false); }, apply);
      }
      // a row's factor: FP64 (g, y) and, for later steps, the reciprocal;
      // FP32 the reciprocal and the right-hand side (a root's x)
      auto put_row = [&](int h, int r, T f, T y, T rr) {
        const int i = rows.slot(r, me + h);
        if constexpr (kYG) {
          if constexpr (kBF) {
            const int q = tab[r] + me + h;
            if (kReuse)
              bf[q].y = y;
            else
              bf[q] = make_double2(f, y);
            if (keep_rcp) rcp_block[q] = rr;
          } else {
            if (!kReuse) sd[i] = f;
            if (keep_rcp) su[i] = rr;
            sb[i] = y;
          }
        } else {
          sd[i] = rr;
          sb[i] = y;
        }
      };
      // FP64: a row's y and the next right-hand side are left for the next
      // row (late_part), where they fill the FP64 pipe while that row's
      // reciprocal, which does not use it, is formed: the chain from pivot to
      // pivot is then the reciprocal and two FP64 instructions.
      constexpr bool kLate = kYG && !kReuse;
      T fp[P], rp[P], bc[P];  // the row before: its factor and reciprocal; this row's right-hand side as given
#pragma unroll
      for (int h = 0; h < P; ++h) fp[h] = rp[h] = bc[h] = T(0);
      auto late_part = [&](int h, int r) {  // of row r - 1
        if (!kLate || r <= first_row[h]) return;
        const T y = B[h] * rp[h];
        B[h] = bc[h] - fp[h] * B[h];
        put_row(h, r - 1, fp[h], y, rp[h]);
      };
      // rows from the distal end: the factor, then the chain to the next row
#pragma unroll kUnroll
      for (int r = 0; r < kL - 1; ++r) {
        if (r < L - 1) {
#pragma unroll
          for (int h = 0; h < P; ++h) {
            if (r < first_row[h]) continue;
            const int i1 = rows.slot(r + 1, me + h);
            const T a1 = sd[i1], b1 = sb[i1], u1 = su[i1];
            if constexpr (kLate) {
              const RcpHalf half = rcp_begin(kCable ? D[h] - uk[h] : D[h]);
              late_part(h, r);
              rp[h] = rcp_end(half);
              fp[h] = uk[h] * rp[h];
              D[h] = a1 - fp[h] * (kCable ? D[h] : uk[h]);
              bc[h] = b1;
            } else {
              const T rr = kReuse ? rk[h] : rcp_solve(D[h]);
              const T f = kReuse ? uk[h] : uk[h] * rr;
              if (!kReuse) D[h] = a1 - f * uk[h];
              const T bn = b1 - f * B[h];
              put_row(h, r, f, kYG ? B[h] * rr : B[h], rr);
              B[h] = bn;
              rk[h] = a1;
            }
            uk[h] = u1;
          }
        }
      }
      // the proximal row, and the contribution to the parent
#pragma unroll
      for (int h = 0; h < P; ++h) {
        if (m.p[h].len == 0) continue;
        const bool root = m.p[h].pcomp < 0;
        const T rr = kReuse ? rk[h] : rcp_solve(kCable && !root ? D[h] - uk[h] : D[h]);
        late_part(h, L - 1);
        const T f = root ? T(0) : kReuse ? uk[h] : uk[h] * rr;  // a cell's root: x = y
        put_row(h, L - 1, f, kYG || root ? B[h] * rr : B[h], rr);
        const T cd = root || kReuse ? T(0) : f * (kCable ? D[h] : uk[h]), cb = root ? T(0) : f * B[h];
        const size_t pos = (size_t)(c0 + me + h);
        slot[2 * pos] = cd;
        slot[2 * pos + 1] = cb;
        cslot[(cur * G::kChunk + me + h) * 2] = cd;
        cslot[(cur * G::kChunk + me + h) * 2 + 1] = cb;
      }
      return;
    }
    T xp[P];
#pragma unroll
    for (int h = 0; h < P; ++h) {
      const Piece& q = m.p[h];
      xp[h] = T(0);
      if (q.len > 0 && q.pcomp >= 0) {
        const int loc = q.ppos - pv.c0;
        xp[h] = (loc >= 0 && loc < pv.n) ? cx[pv.which * G::kChunk + loc] : pre_get(m.xpre[h], T{});
      }
    }
    if constexpr (kYG) {
      // x = y - g x_parent; x goes over g (block order) or over y
      const double2* fb = reinterpret_cast<const double2*>(buf);
      double* sx = reinterpret_cast<double*>(buf);
      auto load = [&](int r, int h) {
        if constexpr (kBF) return fb[tab[r] + me + h];
        const int i = rows.slot(r, me + h);
        return make_double2(sd[i], sb[i]);
      };
      double2 f[P];
#pragma unroll
      for (int h = 0; h < P; ++h) f[h] = load(L - 1, h);
#pragma unroll kUnroll
      for (int r = kL - 1; r >= 0; --r) {
        if (r < L) {
#pragma unroll
          for (int h = 0; h < P; ++h) {
            if (r < first_row[h]) continue;
            const double2 fk = f[h];
            if (r > 0) f[h] = load(r - 1, h);  // (before this row's store)
            const T xi = fk.y - fk.x * xp[h];
            if constexpr (kBF)
              sx[2 * (tab[r] + me + h)] = xi;
            else
              sb[rows.slot(r, me + h)] = xi;
            xp[h] = xi;
          }
        }
      }
    } else {
#pragma unroll kUnroll
      for (int r = kL - 1; r >= 0; --r) {
        if (r < L) {
          const int i = rows.slot(r, me);
#pragma unroll
          for (int h = 0; h < P; ++h) {
            if (r < first_row[h]) continue;
            const T xi = (m.p[h].pcomp < 0 && r == L - 1) ? sb[i + h] : (sb[i + h] - su[i + h] * xp[h]) * sd[i + h];
            sb[i + h] = xi;
            xp[h] = xi;
          }
        }
      }
    }
#pragma unroll
    for (int h = 0; h < P; ++h) {
      if (m.p[h].len == 0) continue;
      static_cast<T*>(Pl.xlast)[c0 + me + h] = xp[h];
      cx[cur * G::kChunk + me + h] = xp[h];
    }
  }

  __device__ static void copy_out(const DevPlan& Pl, const Args& A, int visit, const Meta<P>& m, int n, int lane,
                                  unsigned char* buf) {
    const T* sd = reinterpret_cast<const T*>(buf);
    const T* su = sd + G::kSlots;
    const T* sb = su + G::kSlots;
    const int* tab = reinterpret_cast<const int*>(buf + kTab);
    const long long blk = kPk ? __shfl_sync(kFull, m.p[0].first, 0) : 0;
    if constexpr (kBF) {
      // the elimination wrote its factor block directly; the substitution
      // left x over each slot's g
      if (visit == 0) return;
      const double* sx = reinterpret_cast<const double*>(buf);
      if (kPk) {
        const int e = tab[kL];
#pragma unroll 1
        for (int s = lane; s < e; s += 32) A.x[blk + s] = sx[2 * s];
      } else {
        for_chunk_elements(m, n, lane, [&](int i, int, int row, long long g) { A.x[g] = sx[2 * (tab[row] + i)]; });
      }
      return;
    }
    T* fac = static_cast<T*>(Pl.fac);
    T* rc = reciprocals(Pl);
    const bool keep_fac = visit == 0 && !kReuse, keep_rcp = visit == 0 && keeps_rcp(A);
    if (kPk) {
      const int e = tab[kL];
#pragma unroll 1
      for (int s = lane; s < e; s += 32) {
        if (keep_fac) fac[blk + s] = sd[s];
        if (keep_rcp) rc[blk + s] = su[s];
        A.x[blk + s] = sb[s];
      }
      return;
    }
    for_chunk_elements(m, n, lane, [&](int i, int, int row, long long g) {
      const int q = nidx<P>(row, i);
      if (keep_fac) fac[g] = sd[q];
      if (keep_rcp) rc[g] = su[q];
      A.x[g] = sb[q];
    });
  }
};

// ============================================================================
// Refinement mode (natural layout): one step of iterative refinement on the
// FP32 factor that a FactorMode<float> solve of the same plan left in the
// workspace (the reciprocal pivots).  The elimination visit forms the
// residual r = b - A x of the current x (the FP32 inputs taken exactly;
// products and sums by error-free transformations, so that r keeps FP32
// accuracy although it is tiny next to b) and eliminates it with the stored
// factor, as the FP32 solve eliminated b.  A compartment's residual needs its
// parent's x (the next row; at the proximal row, the parent piece's distal
// compartment) and its children's (the previous row; at a piece's distal
// row, the child pieces pass their products u x up with their
// contributions).  The substitution visit solves for the correction c with
// the same factor and writes x + c.  kIn: x is FP32 (0) or a double-float
// pair (1); kOut: x + c as a pair (0, for another step) or in FP64 (1).
// ============================================================================
template <int P, int kIn, int kOut>
struct RefineMode {
  using V = typename VOf<P>::type;
  using G = Geo<P>;
  static constexpr bool kPacked = false;
  static constexpr bool kNeedsBlk = false;
  static constexpr int kPer = P;
  struct Args {
    const float* d;
    const float* u;
    const float* b;
    const void* x;     // kIn 0: float[n]; 1: float2[n]
    float* rw;         // the eliminated residual (the correction's right-hand side)
    void* xo;          // kOut 0: float2[n]; 1: double[n]
    float* bcorr;      // per piece (branch id): largest |c| of this step
  };
  // staged words: d, u, b (visit 1: the eliminated residual), the factor, and
  // x as pairs (two words per slot; FP32 x uses the first)
  static constexpr int kTab = 6 * G::kSlots * 4;
  static constexpr int kStageBytes = kTab + 96;
  static constexpr int kCslot = 0, kCx = 0, kCacheBytes = 2 * G::kChunk * 16;
  static constexpr int kTeamBytes = 2 * kStageBytes + kCacheBytes;
  static constexpr int kWarpBytes = kStageBytes + kCacheBytes;
  static constexpr int kMinBlocks = teams_per_sm(kTeamBytes, 10), kMinBlocksAlone = teams_per_sm(2 * kWarpBytes, 10);
  // the same, by stretch only (one step: 1.0 82 : 107, 1.22 727 : 802, 1.31 1042
  // : 1235, 1.5 2065 : 2447, 886 : 886 and 202 : 194, 1.9 2008 : 2019, 2.0 1727 :
  // 1317)
  static constexpr int kTeamShare = 1 << 20;
  static constexpr double kTeamSpeed = 1.6;
  __device__ static void init_buffer(unsigned char*) {}

  // what the chunk needs of earlier chunks: the parent's x (visit 0), the
  // parent's correction where no cache holds it (visit 1)
  template <bool kAlone>
  __device__ static void fetch(const DevPlan& Pl, const Args& A, int visit, Meta<P>& m, const Prev& pv) {
#pragma unroll
    for (int h = 0; h < P; ++h) {
      const Piece& q = m.p[h];
      if (q.len == 0 || q.pcomp < 0) continue;
      const int loc = q.ppos - pv.c0;
      if (visit == 0)
        m.xpre[h].ff = gx(A, q.pcomp);
      else if (!(loc >= 0 && loc < pv.n))
        m.xpre[h].f = static_cast<const float2*>(Pl.xlast)[q.ppos].x;
    }
  }

  __device__ static void stage(const DevPlan& Pl, const Args& A, int visit, const Meta<P>& m, int n, int lane,
                               unsigned char* buf) {
    float* sd = reinterpret_cast<float*>(buf);
    float* su = sd + G::kSlots;
    float* sb = su + G::kSlots;
    float* sf = sb + G::kSlots;
    float* sx = sf + G::kSlots;  // [2 * kSlots]
    const float* fac = static_cast<const float*>(Pl.fac);
    for_chunk_elements(m, n, lane, [&](int i, int, int row, long long g) {
      const int q = nidx<P>(row, i);
      if (visit == 0) {
        cp_async4(&sd[q], A.d + g);
        cp_async4(&sb[q], A.b + g);
      } else {
        cp_async4(&sb[q], A.rw + g);
      }
      cp_async4(&su[q], A.u + g);
      cp_async4(&sf[q], fac + g);
      if (kIn == 1)
        cp_async8(&sx[2 * q], static_cast<const float2*>(A.x) + g);
      else
        cp_async4(&sx[2 * q], static_cast<const float*>(A.x) + g);
    });
    cp_commit();
  }

  // x of a row: the lane's P values as a double-float pair
  __device__ static FFV<V> ldx(const float* sx, int idx) {
    if constexpr (P == 2) {
      const float4 v = *reinterpret_cast<const float4*>(sx + 2 * idx);
      return {f2_make(v.x, v.z), kIn == 1 ? f2_make(v.y, v.w) : f2_make(0.f, 0.f)};
    } else {
      const float2 v = *reinterpret_cast<const float2*>(sx + 2 * idx);
      return {v.x, kIn == 1 ? v.y : 0.f};
    }
  }
  // x of a compartment in global memory (a parent's distal compartment)
  __device__ static float2 gx(const Args& A, long long g) {
    if (kIn == 1) return static_cast<const float2*>(A.x)[g];
    return make_float2(static_cast<const float*>(A.x)[g], 0.f);
  }
  // acc -= t, accumulating the rounding errors of the leading parts exactly
  // (two-sum) and everything else in the second word
  __device__ static void acc_sub(V& s, V& e, const FFV<V>& t) {
    const V s1 = vsub(s, t.h);
    const V bb = vsub(s1, s);
    const V err = vsub(vsub(s, vsub(s1, bb)), vadd(t.h, bb));
    e = vadd(e, vsub(err, t.l));
    s = s1;
  }

  template <bool kAlone>
  __device__ static void compute(const DevPlan& Pl, const Args& A, int visit, int c0, int n, int lane,
                                 const Meta<P>& m, unsigned char* buf, const Prev& pv, unsigned char* cache, int cur) {
    float* sd = reinterpret_cast<float*>(buf);
    float* su = sd + G::kSlots;
    float* sb = su + G::kSlots;
    float* sf = sb + G::kSlots;
    float* sx = sf + G::kSlots;
    float4* cslot = reinterpret_cast<float4*>(cache + kCslot);  // [2][kChunk] (u x up, eliminated residual up)
    float* cx = reinterpret_cast<float*>(cache + kCx);          // [2][kChunk] distal corrections
    float4* slot = static_cast<float4*>(Pl.cd);
    float2* xlast = static_cast<float2*>(Pl.xlast);
    const int L = m.L;
    const unsigned live = kAlone ? __ballot_sync(kFull, L > 0) : 0u;  // (for_children)
    if (L == 0) return;
    const int me = P * lane;
    const int delta = P == 2 ? L - m.p[P - 1].len : 0;
    // a cell's root has no parent: its coupling is not part of the system
#pragma unroll
    for (int h = 0; h < P; ++h)
      if (m.p[h].len > 0 && m.p[h].pcomp < 0) su[nidx<P>(L - 1, me + h)] = 0.f;
    if (visit == 0) {
      // per piece: the parent's x, and the children's u x and eliminated residuals
      float xph[P], xpl[P], crh[P], crl[P], ce[P];
#pragma unroll
      for (int h = 0; h < P; ++h) {
        const Piece& q = m.p[h];
        xph[h] = xpl[h] = crh[h] = crl[h] = ce[h] = 0.f;
        if (!kAlone && q.len == 0) continue;  // (a lone warp's lanes go on together)
        if (q.len > 0 && q.pcomp >= 0) {
          const float2 t = m.xpre[h].ff;
          xph[h] = t.x;
          xpl[h] = t.y;
        }
        ff acc = {0.f, 0.f};
        for_children<kAlone>(
            live, q.nchild, 0,
            [&](int c) {
              const int cp = child_pos(Pl, q, c);
              const int loc = cp - pv.c0;
              return (loc >= 0 && loc < pv.n) ? cslot[pv.which * G::kChunk + loc] : slot_load(slot + cp, q);
            },
            [&](const float4& v) {
              acc = ff_sub(acc, -v.x, -v.y);
              ce[h] += v.z;
            });
        crh[h] = acc.h;
        crl[h] = acc.l;
      }
      FFV<V> tc{vpack<P>(crh), vpack<P>(crl)};  // the children's u x (at a distal row), or the chain child's
      V cev = vpack<P>(ce);                    // the children's eliminated residuals times their multipliers
      FFV<V> un{}, en{};                       // the proximal row's u x and eliminated residual times multiplier
#pragma unroll
      for (int r = 0; r < kL; ++r) {
        if (r < L) {
          if constexpr (P == 2) {
            if (r > 0 && r == delta) {
              tc = {vset_hi(tc.h, crh[1]), vset_hi(tc.l, crl[1])};
              cev = vset_hi(cev, ce[1]);
            }
          }
          const int i = nidx<P>(r, me);
          const V dk = ldv(sd, i, V{}), uk = ldv(su, i, V{}), bk = ldv(sb, i, V{}), fk = ldv(sf, i, V{});
          const FFV<V> xk = ldx(sx, i);
          FFV<V> xn;
          if (r < L - 1)
            xn = ldx(sx, nidx<P>(r + 1, me));
          else
            xn = {vpack<P>(xph), vpack<P>(xpl)};
          V s = bk, e = vsplat(0.f, V{});
          acc_sub(s, e, vmul_f(xk, dk));
          acc_sub(s, e, vmul_f(xn, uk));
          acc_sub(s, e, tc);
          const V rp = vsub(vadd(s, e), cev);  // the residual, less the children's eliminated residuals
          stv(sb, i, rp);
          tc = vmul_f(xk, uk);                 // this row's u x, for the next row (or the parent)
          cev = vmul(vmul(uk, fk), rp);        // multiplier u / pivot times the eliminated residual
          un = tc;
          en = {cev, vsplat(0.f, V{})};
        }
      }
#pragma unroll
      for (int h = 0; h < P; ++h) {
        if (m.p[h].len == 0) continue;
        const float4 out = m.p[h].pcomp >= 0 ? make_float4(vget(un.h, h), vget(un.l, h), vget(en.h, h), 0.f)
                                             : make_float4(0.f, 0.f, 0.f, 0.f);
        slot[c0 + me + h] = out;
        cslot[cur * G::kChunk + me + h] = out;
      }
      return;
    }
    // the correction from the proximal row down, and x + c
    float cph[P];
#pragma unroll
    for (int h = 0; h < P; ++h) {
      const Piece& q = m.p[h];
      cph[h] = 0.f;
      if (q.len > 0 && q.pcomp >= 0) {
        const int loc = q.ppos - pv.c0;
        cph[h] = (loc >= 0 && loc < pv.n) ? cx[pv.which * G::kChunk + loc] : m.xpre[h].f;
      }
    }
    V cp = vpack<P>(cph);
    float cm[P], cb = 0.f;
#pragma unroll
    for (int h = 0; h < P; ++h) cm[h] = 0.f;
#pragma unroll
    for (int r = kL - 1; r >= 0; --r) {
      if (r < L) {
        const int i = nidx<P>(r, me);
        const V uk = ldv(su, i, V{}), rk = ldv(sb, i, V{}), fk = ldv(sf, i, V{});
        const V c = vmul(vfma(vneg(uk), cp, rk), fk);
        const FFV<V> xk = ldx(sx, i);
        // x + c: two-sum of the leading parts, the rest into the low word
        const V s = vadd(xk.h, c);
        const V bb = vsub(s, xk.h);
        const V err = vadd(vsub(xk.h, vsub(s, bb)), vsub(c, bb));
        const FFV<V> xn = vrenorm(s, vadd(err, xk.l));
#pragma unroll
        for (int h = 0; h < P; ++h) {
          const int q = i + h;
          if (r >= L - m.p[h].len) cm[h] = fmaxf(cm[h], fabsf(vget(c, h)));
          if (kOut == 1)
            reinterpret_cast<double*>(sx)[q] = ff_to_double(vget(xn.h, h), vget(xn.l, h));
          else
            reinterpret_cast<float2*>(sx)[q] = make_float2(vget(xn.h, h), vget(xn.l, h));
        }
        if constexpr (P == 2) {
          if (r == delta) cb = f2_hi(c);
        }
        cp = c;
      }
    }
#pragma unroll
    for (int h = 0; h < P; ++h) {
      if (m.p[h].len == 0) continue;
      const float cd = h == 0 ? vget(cp, 0) : cb;
      const int pos = c0 + me + h;
      xlast[pos] = make_float2(cd, 0.f);
      cx[cur * G::kChunk + me + h] = cd;
      if (A.bcorr) A.bcorr[Pl.pos_branch[pos]] = cm[h];
    }
  }

  __device__ static void copy_out(const DevPlan&, const Args& A, int visit, const Meta<P>& m, int n, int lane,
                                  unsigned char* buf) {
    const float* sd = reinterpret_cast<const float*>(buf);
    const float* sb = sd + 2 * G::kSlots;
    const float* sx = sd + 4 * G::kSlots;
    for_chunk_elements(m, n, lane, [&](int i, int, int row, long long g) {
      const int q = nidx<P>(row, i);
      if (visit == 0)
        A.rw[g] = sb[q];
      else  // (an FP64 x as its two words)
        static_cast<float2*>(A.xo)[g] = reinterpret_cast<const float2*>(sx)[q];
    });
  }
};

// ============================================================================
// Task driver
// ============================================================================
// Position in a task's chunk sequence: chunks deepest-first for the
// elimination (visit 0), root-side first for the substitution (visit 1).
struct Pos {
  int visit, l, c0, n;  // visit == ve: past the end
};

// The task's chunk boundaries (nl + 1 positions): a window of 32 of them is
// held one per lane, so that stepping to the next chunk is two shuffles
// instead of two dependent loads.
struct ChunkTable {
  const int32_t* lp;
  int nl, w, v;
  __device__ __forceinline__ ChunkTable(const int32_t* lp_, int nl_) : lp(lp_), nl(nl_), w(-64), v(0) {}
  __device__ __forceinline__ Pos at(int visit, int l, int lane) {
    if (l < w || l + 1 > w + 31) {
      w = visit == 0 ? (l > 30 ? l - 30 : 0) : l;
      v = w + lane <= nl ? __ldg(lp + w + lane) : 0;
    }
    const int c0 = __shfl_sync(kFull, v, l - w);
    return {visit, l, c0, __shfl_sync(kFull, v, l + 1 - w) - c0};
  }
  __device__ __forceinline__ Pos next(const Pos& p, int ve, int lane) {
    if (p.visit == 0) {
      if (p.l > 0) return at(0, p.l - 1, lane);
      if (ve == 1) return {ve, 0, 0, 0};
      return at(1, 0, lane);
    }
    if (p.l + 1 < nl) return at(1, p.l + 1, lane);
    return {ve, 0, 0, 0};
  }
};

// One task by a team.  Per step, between two barriers of the CTA, warp 0
// computes chunk k while warp 1 copies out the results of chunk k - 1 and
// stages chunk k + 1 into the same buffer: the two warps meet only at the
// barrier, and neither waits for anything else.  Where the sweeps turn, the
// first chunk of the substitution is staged only after the last one of the
// elimination is out (it is the same chunk, and reads what the elimination
// left).  In one warp with one buffer (run_task_alone) a chunk of the natural
// compensated solve took 17.4k clocks in the elimination, 8.9k of them
// arithmetic, and 13.1k in the substitution, 5.4k of them arithmetic.  Against
// lone warps: FP64 solve of 64 small cells 47.1 -> 41.0 us, FP32 solve of 1001
// small cells 79 -> 64 us, 40-step rollout with gradients 27.9 -> 22.5 ms, two
// refinement steps 2.16 -> 1.88 ms, host pipeline 3.12 -> 2.66 ms.  Loops over
// a chunk's elements stay rolled: code that overruns the instruction cache
// costs more than their bookkeeping (solve of 28M compartments 835 -> 789 us
// without the compiler's unrolling, 958 us with four steps at a time).
template <class M>
__device__ void run_task(const DevPlan& Pl, const typename M::Args& A, const TaskRec& t, bool mover, int lane,
                         unsigned char* smem) {
  constexpr int P = M::kPer;
  ChunkTable tab(Pl.tlvl_ptr + t.lvl_off, t.nlvl);
  const int vb = t.code == 2 ? 1 : 0, ve = t.code == 1 ? 1 : 2;
  unsigned char* cache = smem + 2 * M::kStageBytes;
  auto buf = [smem](int which) { return smem + which * M::kStageBytes; };
  auto meta = [&](const Pos& p) { return load_meta<M::kPacked, P>(Pl, p.c0, p.n, lane, M::kNeedsBlk); };
  auto stage = [&](const Pos& p, const Meta<P>& m, int which) {
    M::stage(Pl, A, p.visit, m, p.n, lane, buf(which));
    cp_wait_all();
  };
  // metadata runs two chunks ahead
  Pos cur = tab.at(vb, vb == 0 ? t.nlvl - 1 : 0, lane);
  Meta<P> m_cur = unpack_meta(meta(cur)), m_prev = m_cur;
  Pos nxt = tab.next(cur, ve, lane);
  const RawMeta<M::kPacked, P> r_nxt = meta(nxt);
  Prev pv{0, 0, 0};  // the chunk before, if of the same sweep
  if (mover)
    stage(cur, m_cur, 0);
  else
    M::template fetch<false>(Pl, A, cur.visit, m_cur, pv);
  Meta<P> m_nxt = unpack_meta(r_nxt);
  int which = 0;
  __syncthreads();
  for (;;) {
    const bool turn = nxt.visit != cur.visit;  // the last chunk of a sweep
    const Prev pn = turn ? Prev{0, 0, 0} : Prev{cur.c0, cur.n, cur.l & 1};
    const Pos nn = nxt.visit < ve ? tab.next(nxt, ve, lane) : nxt;
    const RawMeta<M::kPacked, P> r_nn = meta(nn);
    if (mover) {
      if (pv.n > 0) M::copy_out(Pl, A, cur.visit, m_prev, pv.n, lane, buf(which ^ 1));
      __syncwarp();
      if (!turn) stage(nxt, m_nxt, which ^ 1);
    } else {
      if (!turn) M::template fetch<false>(Pl, A, nxt.visit, m_nxt, pn);
      M::template compute<false>(Pl, A, cur.visit, cur.c0, cur.n, lane, m_cur, buf(which), pv, cache, cur.l & 1);
      __syncwarp();
      if (turn) {  // this warp's factors and contributions, for bulk copies and other teams
        __threadfence();
        fence_async();
      }
    }
    __syncthreads();
    if (turn) {
      const bool done = nxt.visit >= ve;
      if (mover) {
        M::copy_out(Pl, A, cur.visit, m_cur, cur.n, lane, buf(which));
        __threadfence();
        fence_async();
        __syncwarp();
        if (!done) stage(nxt, m_nxt, which ^ 1);
      } else if (!done) {
        M::template fetch<false>(Pl, A, nxt.visit, m_nxt, pn);
      }
      __syncthreads();
      if (done) return;
    }
    pv = pn;
    m_prev = m_cur;
    cur = nxt;
    m_cur = m_nxt;
    nxt = nn;
    m_nxt = unpack_meta(r_nn);
    which ^= 1;
  }
}

// The same by one warp with one staging buffer: more tasks at a time, for
// launches that have them.
template <class M>
__device__ void run_task_alone(const DevPlan& Pl, const typename M::Args& A, const TaskRec& t, int lane,
                               unsigned char* smem) {
  constexpr int P = M::kPer;
  ChunkTable tab(Pl.tlvl_ptr + t.lvl_off, t.nlvl);
  const int vb = t.code == 2 ? 1 : 0, ve = t.code == 1 ? 1 : 2;
  unsigned char* cache = smem + M::kStageBytes;
  auto meta = [&](const Pos& p) { return load_meta<M::kPacked, P>(Pl, p.c0, p.n, lane, M::kNeedsBlk); };
  Pos cur{vb, 0, 0, 0}, nxt = tab.at(vb, vb == 0 ? t.nlvl - 1 : 0, lane);
  Meta<P> m_cur = unpack_meta(meta(nxt)), m_nxt = m_cur;
  Prev pv{0, 0, 0}, pn{0, 0, 0};
  while (nxt.visit < ve) {
    if (nxt.visit != cur.visit) {  // this warp's elimination, for the substitution's bulk copies
      __threadfence();
      fence_async();
      __syncwarp();
    }
    cur = nxt;
    m_cur = m_nxt;
    pv = pn;
    M::stage(Pl, A, cur.visit, m_cur, cur.n, lane, smem);
    M::template fetch<true>(Pl, A, cur.visit, m_cur, pv);
    nxt = tab.next(cur, ve, lane);
    const RawMeta<M::kPacked, P> r_nxt = meta(nxt);
    cp_wait_all();
    __syncwarp();
    M::template compute<true>(Pl, A, cur.visit, cur.c0, cur.n, lane, m_cur, smem, pv, cache, cur.l & 1);
    __syncwarp();
    M::copy_out(Pl, A, cur.visit, m_cur, cur.n, lane, smem);
    __syncwarp();
    pn = nxt.visit != cur.visit ? Prev{0, 0, 0} : Prev{cur.c0, cur.n, cur.l & 1};
    m_nxt = unpack_meta(r_nxt);
  }
  __threadfence();  // (a hand-over follows)
  __syncwarp();
}

// After a subtree task's elimination: count its units as done; whoever
// finishes the cell's last subtree takes over the cell's top part (both
// visits) as its next task.  Nothing waits: the hand-over goes to whoever
// arrives last.  One thread; returns the top task, or -1.  Release: every lane fenced
// its writes before the team's last barrier (a lone warp's __syncwarp), which
// this thread passed.  Acquire: this thread's fence after the atomic reaches
// the other lanes of a team through the team's next barrier; a lone warp's
// lanes, which learn of the top part by a shuffle (no memory ordering), fence
// themselves (k_units).  The top part reads those slots through L2.
__device__ __forceinline__ int hand_over(const DevPlan& P, int t) {
  const int cell = __ldg(P.task_sub + 2 * t);
  if (cell < 0) return -1;
  const int cnt = __ldg(P.task_sub + 2 * t + 1);
  __threadfence();
  if (atomicAdd(P.cell_done + cell, cnt) + cnt != __ldg(P.cell_nsub + cell)) return -1;
  P.counter[2] = 0;  // (phase C's, launch_phases)
  __threadfence();
  return __ldg(P.cell_top_task + cell);
}

// kTeam: a CTA is one team; else its two warps run a task each.
template <class M, bool kTeam>
__host__ __device__ constexpr int cta_bytes() {
  return kTeam ? M::kTeamBytes + 16 : 2 * M::kWarpBytes;
}
template <class M, bool kTeam>
__global__ void __launch_bounds__(64, kTeam ? M::kMinBlocks : M::kMinBlocksAlone)
    k_units(DevPlan P, typename M::Args A, int phase) {
  extern __shared__ __align__(16) unsigned char smem_u[];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int* ctl = reinterpret_cast<int*>(smem_u + M::kTeamBytes);  // the team's next entry, or top part
  constexpr int kWarpBytes = cta_bytes<M, kTeam>() / 2;
  unsigned char* smem = kTeam ? smem_u : smem_u + w * kWarpBytes;
  bool mover = false;
  if (kTeam) {
    if (threadIdx.x < 2) M::init_buffer(smem_u + threadIdx.x * M::kStageBytes);
    __syncthreads();
    mover = w == 1;
  } else {
    if (lane == 0) M::init_buffer(smem);
    __syncwarp();
  }
  const int e0 = P.phase_off[phase], ne = P.phase_off[phase + 1] - e0;
  const int runners = kTeam ? (int)gridDim.x : 2 * (int)gridDim.x;
  int* next_entry = P.counter + phase;
  auto entry = [&](int i) {
    const int4 r = __ldg(P.phase_rec + e0 + i);
    return TaskRec{(uint32_t)r.x, r.y, r.z, r.w};
  };
  // the first entry of a runner (team or warp) is its own number, the others
  // are counted off
  int k = kTeam ? (int)blockIdx.x : 2 * (int)blockIdx.x + w;
  TaskRec t = entry(k < ne ? k : 0);
  while (k < ne) {  // (one warp of the last CTA, at most, has no entry)
    if constexpr (kTeam)
      run_task<M>(P, A, t, mover, lane, smem);
    else
      run_task_alone<M>(P, A, t, lane, smem);
    // the next entry: a top part handed over (-2 - task), or one counted off
    if (kTeam ? threadIdx.x == 0 : lane == 0) {
      const int top = t.code == 1 ? hand_over(P, t.id) : -1;
      k = top >= 0 ? -2 - top : ne <= runners ? ne : runners + atomicAdd(next_entry, 1);
      if (kTeam) ctl[0] = k;
    }
    if constexpr (kTeam) {
      __syncthreads();
      k = ctl[0];
      __syncthreads();
    } else {
      k = __shfl_sync(kFull, k, 0);
      if (k < 0) {  // a top part: every lane's side of the acquire (hand_over)
        __threadfence();
        __syncwarp();
      }
    }
    if (k >= ne) break;
    t = k >= 0 ? entry(k) : TaskRec{(uint32_t)P.task_lvl_off[-2 - k], P.task_nlvl[-2 - k], -2 - k, 0};
  }
  if (phase == 2) {  // phase A's counts back to 0 (launch_phases)
    if (blockIdx.x == 0 && threadIdx.x == 0) P.counter[0] = 0;
    for (int c = blockIdx.x * 64 + threadIdx.x; c < P.n_cells; c += gridDim.x * 64) P.cell_done[c] = 0;
  }
}

template <class M, bool kTeam>
cudaError_t grid_of(const DevPlan& P, int* grid) {
  int per_sm = 0;
  const size_t smem = cta_bytes<M, kTeam>();
  const auto kernel = k_units<M, kTeam>;
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, 64, smem);
  if (e != cudaSuccess) return e;
  *grid = P.sms * (per_sm > 0 ? per_sm : 1);
  return cudaSuccess;
}
// persistent grid sizes of both kernels of a mode: teams, and CTAs of two lone warps
template <class M>
cudaError_t grid_of(const DevPlan& P, RunnerGrid* grid) {
  cudaError_t e = grid_of<M, true>(P, &grid->teams);
  return e == cudaSuccess ? grid_of<M, false>(P, &grid->ctas) : e;
}

// The work counters and the cells' counts of finished subtrees are 0 when they
// are needed without a copy before each call: phase C's launch zeroes phase
// A's counter and every cell's count for the next call, phase A's hand-overs
// zero phase C's counter, whatever they hold.  Where no cell is cut there is no phase C, and a memset follows phase A
// if it counted entries off at all (FP64 solve of 59M compartments 1541.7 us
// with and without).
// So even calls that share a plan unordered, against the interface, leave sound
// counts once they have all ended: each call's zeroing comes after its own
// counting, hence the last zeroing after all of it.  (Restored by whoever drew
// the last entry or finished the last subtree, a count that once went wrong
// stayed wrong, and later calls left out entries or top parts silently.)
template <class M>
cudaError_t launch_phases(const DevPlan& P, const typename M::Args& A, const RunnerGrid& grid, cudaStream_t s) {
  if (P.n_wtasks == 0) return cudaSuccess;
  const bool cut = P.phase_off[3] > P.phase_off[2];
  for (int phase = 0; phase < 3; ++phase) {
    const int ne = P.phase_off[phase + 1] - P.phase_off[phase];
    if (ne == 0) continue;
    int runners;
    // Teams where one warp per entry leaves the chip idle anyway or a task's
    // own latency decides, lone warps, twice as many tasks at a time, where
    // there are entries for them.  Phase A ends with the longest chains of
    // chunks, so more entries than teams may still do better on teams: up to
    // the mode's share, and while phase A on the fewer teams is not longer, in
    // chunks, than a team is faster at a chunk (RunnerGrid::stretch, the
    // mode's kTeamSpeed).  Without the second bound 2000 equal tasks ran on 1216
    // or 1824 teams in two rounds where lone warps take one: 2000 stars of 3000
    // compartments FP64 3.22 ms, by lone warps 1.79, compensated 2.60 and 1.52;
    // a million cells of 12 compartments 731 and 536, 501 and 399 us.  Phase C
    // (subtrees' substitutions) has no such tail: teams while every entry has
    // one (2306 entries on 1824 teams 263 us, on lone warps 214).
    const bool teams = phase == 0 ? (int64_t)ne * 16 <= (int64_t)M::kTeamShare * grid.teams &&
                                        grid.stretch <= M::kTeamSpeed
                                  : ne <= grid.teams;
    if (teams) {
      runners = ne < grid.teams ? ne : grid.teams;
      k_units<M, true><<<runners, 64, cta_bytes<M, true>(), s>>>(P, A, phase);
    } else {
      const int ctas = (ne + 1) / 2 < grid.ctas ? (ne + 1) / 2 : grid.ctas;
      runners = 2 * ctas;
      k_units<M, false><<<ctas, 64, cta_bytes<M, false>(), s>>>(P, A, phase);
    }
    cudaError_t e = cudaGetLastError();
    if (e == cudaSuccess && !cut && ne > runners) e = cudaMemsetAsync(P.counter, 0, 4 * sizeof(int32_t), s);
    if (e != cudaSuccess) {
      cudaMemsetAsync(P.counter, 0, ((size_t)P.n_cells + 4) * sizeof(int32_t), s);
      return e;
    }
  }
  return cudaSuccess;
}

// ---- the modes' instantiations for P pieces per lane --------------------------
template <int PL>
struct UnitKernels {
  using F64 = FactorMode<double, false, false, PL>;
  using F32 = FactorMode<float, false, false, PL>;
  using Cable = FactorMode<double, true, false, PL>;
  using Comp = CompMode<false, PL>;
  using PkF64 = FactorMode<double, false, true, PL>;
  using PkF32 = FactorMode<float, false, true, PL>;
  using PkComp = CompMode<true, PL>;
  using PkCable = FactorMode<double, true, true, PL>;
  using CableReuse = FactorMode<double, true, false, PL, true>;
  using PkCableReuse = FactorMode<double, true, true, PL, true>;
  // the FP64 kinds with the factor at natural positions (small batches)
  using F64N = FactorMode<double, false, false, PL, false, false>;
  using CableN = FactorMode<double, true, false, PL, false, false>;
  using PkF64N = FactorMode<double, false, true, PL, false, false>;
  using PkCableN = FactorMode<double, true, true, PL, false, false>;
  using CableReuseN = FactorMode<double, true, false, PL, true, false>;
  using PkCableReuseN = FactorMode<double, true, true, PL, true, false>;
  using R32to2 = RefineMode<PL, 0, 0>;
  using R32to64 = RefineMode<PL, 0, 1>;
  using R2to2 = RefineMode<PL, 1, 0>;
  using R2to64 = RefineMode<PL, 1, 1>;

  static cudaError_t prepare(DevPlan& P) {
    cudaError_t e = grid_of<F64>(P, &P.grid[0]);
    if (e == cudaSuccess) e = grid_of<F32>(P, &P.grid[1]);
    if (e == cudaSuccess) e = grid_of<Cable>(P, &P.grid[2]);
    if (e == cudaSuccess) e = grid_of<Comp>(P, &P.grid[3]);
    if (e == cudaSuccess) e = grid_of<PkF64>(P, &P.grid[4]);
    if (e == cudaSuccess) e = grid_of<PkF32>(P, &P.grid[5]);
    if (e == cudaSuccess) e = grid_of<PkComp>(P, &P.grid[6]);
    if (e == cudaSuccess) e = grid_of<PkCable>(P, &P.grid[7]);
    RunnerGrid g_reuse;  // same footprint as the plain modes
    if (e == cudaSuccess) e = grid_of<CableReuse>(P, &g_reuse);
    if (e == cudaSuccess) e = grid_of<PkCableReuse>(P, &g_reuse);
    if (e == cudaSuccess) e = grid_of<R32to2>(P, &P.grid_refine);
    if (e == cudaSuccess) e = grid_of<R32to64>(P, &g_reuse);
    if (e == cudaSuccess) e = grid_of<R2to2>(P, &g_reuse);
    if (e == cudaSuccess) e = grid_of<R2to64>(P, &g_reuse);
    if (e == cudaSuccess) e = grid_of<F64N>(P, &P.grid_nf[0]);
    if (e == cudaSuccess) e = grid_of<CableN>(P, &P.grid_nf[1]);
    if (e == cudaSuccess) e = grid_of<PkF64N>(P, &P.grid_nf[2]);
    if (e == cudaSuccess) e = grid_of<PkCableN>(P, &P.grid_nf[3]);
    if (e == cudaSuccess) e = grid_of<CableReuseN>(P, &g_reuse);
    if (e == cudaSuccess) e = grid_of<PkCableReuseN>(P, &g_reuse);
    return e;
  }

  static cudaError_t run(const DevPlan& P, const UnitCall& c, cudaStream_t s) {
    const double* d8 = static_cast<const double*>(c.d);
    const double* u8 = static_cast<const double*>(c.u);
    const double* s8 = static_cast<const double*>(c.s);
    const double* g8 = static_cast<const double*>(c.g);
    double* x8 = static_cast<double*>(c.x);
    const float* d4 = static_cast<const float*>(c.d);
    const float* u4 = static_cast<const float*>(c.u);
    const float* b4 = static_cast<const float*>(c.b);
    float* x4 = static_cast<float*>(c.x);
    const double th = (double)c.theta;
    const bool blk = P.fp64_blocks != 0;
    switch (c.op) {
      case UnitOp::F64:
        if (!blk) return launch_phases<F64N>(P, {d8, u8, nullptr, nullptr, x8, 0.0, 0.0, 0.0, false}, P.grid_nf[0], s);
        return launch_phases<F64>(P, {d8, u8, nullptr, nullptr, x8, 0.0, 0.0, 0.0, false}, P.grid[0], s);
      case UnitOp::F32:
        return launch_phases<F32>(P, {d4, u4, nullptr, nullptr, x4, 0.f, 0.f, 0.f, false,
                                      static_cast<const float*>(c.rhs)}, P.grid[1], s);
      case UnitOp::Comp:
        return launch_phases<Comp>(P, {d4, u4, b4, x8}, P.grid[3], s);
      case UnitOp::Cable:
        if (!blk)
          return launch_phases<CableN>(P, {nullptr, u8, s8, g8, x8, c.dt, c.E, th, c.rhs_from_V}, P.grid_nf[1], s);
        return launch_phases<Cable>(P, {nullptr, u8, s8, g8, x8, c.dt, c.E, th, c.rhs_from_V}, P.grid[2], s);
      case UnitOp::CableReuse:
        if (!blk) return launch_phases<CableReuseN>(P, {nullptr, u8, s8, g8, x8, c.dt, c.E, th, true}, P.grid_nf[1], s);
        return launch_phases<CableReuse>(P, {nullptr, u8, s8, g8, x8, c.dt, c.E, th, true}, P.grid[2], s);
      case UnitOp::PkF64:
        if (!blk)
          return launch_phases<PkF64N>(P, {d8, u8, nullptr, nullptr, x8, 0.0, 0.0, 0.0, false}, P.grid_nf[2], s);
        return launch_phases<PkF64>(P, {d8, u8, nullptr, nullptr, x8, 0.0, 0.0, 0.0, false}, P.grid[4], s);
      case UnitOp::PkF32:
        return launch_phases<PkF32>(P, {d4, u4, nullptr, nullptr, x4, 0.f, 0.f, 0.f, false}, P.grid[5], s);
      case UnitOp::PkComp:
        return launch_phases<PkComp>(P, {d4, u4, b4, x8}, P.grid[6], s);
      case UnitOp::PkCable:
        if (!blk)
          return launch_phases<PkCableN>(P, {nullptr, u8, s8, g8, x8, c.dt, c.E, th, c.rhs_from_V}, P.grid_nf[3], s);
        return launch_phases<PkCable>(P, {nullptr, u8, s8, g8, x8, c.dt, c.E, th, c.rhs_from_V}, P.grid[7], s);
      case UnitOp::PkCableReuse:
        if (!blk)
          return launch_phases<PkCableReuseN>(P, {nullptr, u8, s8, g8, x8, c.dt, c.E, th, true}, P.grid_nf[3], s);
        return launch_phases<PkCableReuse>(P, {nullptr, u8, s8, g8, x8, c.dt, c.E, th, true}, P.grid[7], s);
      case UnitOp::Refine32to2:
        return launch_phases<R32to2>(P, {d4, u4, b4, c.rhs, c.rw, c.x, c.bcorr}, P.grid_refine, s);
      case UnitOp::Refine32to64:
        return launch_phases<R32to64>(P, {d4, u4, b4, c.rhs, c.rw, c.x, c.bcorr}, P.grid_refine, s);
      case UnitOp::Refine2to2:
        return launch_phases<R2to2>(P, {d4, u4, b4, c.rhs, c.rw, c.x, c.bcorr}, P.grid_refine, s);
      case UnitOp::Refine2to64:
        return launch_phases<R2to64>(P, {d4, u4, b4, c.rhs, c.rw, c.x, c.bcorr}, P.grid_refine, s);
    }
    return cudaErrorInvalidValue;
  }
};

}  // namespace
}  // namespace hines
