// bfs_block.cuh -- the 2BFS pseudo-diameter of Sec. 6 run by ONE block: for
// the teams of the batched and serving kernels, and for small systems.
//
// The group version (bfs_core.cuh) pays, per BFS level, a group barrier and a
// chain of global-memory round trips (queue size, queue entry, row pointers,
// columns, the claim on dist, the queue counter).  Here a single block runs
// both searches with block barriers, visited BITMAPS (a claim is one atomicOr
// on a bit), one frontier queue for both searches (entries tagged with their
// search) and its counters in shared memory.  What bounds a level is its
// chain of dependent loads, so the neighbours are read from the sliced layout
// whose slice offsets are kept in shared memory: one global round trip a
// level instead of two (row pointers, then columns).
//
// Storage (given by the caller), by what fits the block's buffer:
//   * both bitmaps and the slice offsets (3 n / 8 bytes): one round trip a level;
//   * both bitmaps (n / 4 bytes): neighbours from the caller's CSR;
//   * one bitmap: the searches run one after the other;
//   * else bitmaps in global scratch.
// The queues take the rest of the buffer, and entries past that capacity go
// to global queues.  So any n works; shared memory only makes it faster.  A
// matrix with a row longer than the sliced layout keeps uses the CSR.
//
// Readings are those of bfs_core.cuh: search A from vertex 0; t = smallest
// vertex at the largest distance from 0 = smallest vertex of A's last
// non-empty level; l~ = last non-empty level of the BFS from t; the search
// from t is started speculatively from n - 1 with A.  Unlike the group
// version, B is dropped as soon as A ends with t != n - 1.  Only connected
// graphs are handled; otherwise the caller runs the group version.
#pragma once
#include <limits.h>

#include "common.cuh"

namespace mpcg {

// The graph as the block search reads it.
struct BlockGraph {
  const int32_t* rp;
  const int32_t* col;
  const int32_t* slice_ptr;
  const uint32_t* slice_w;
  const void* scol;  // sliced columns: int16 offsets from the row (c16) or int32
  int n, c16;
};

struct BlockBfs {
  BlockGraph g;
  uint32_t *visA, *visB;  // visited bitmaps of searches A and B, (n + 31) / 32 words each
  const int32_t* sp;   // slice offsets in shared memory, or null: the CSR is read
  int32_t* qs;         // shared queue heads: even levels, then odd levels (cap entries each)
  int32_t *qg0, *qg1, *qg2, *qg3;  // global queues of n entries: even levels 0 and 1, odd 2 and 3
  int cap;
  bool dual;           // both searches at once (two bitmaps)
  int* cnt;            // shared: queue sizes [0..2] and B's part of them [3..5] by level
                       // mod 3, [6] scratch, [7] set when the search is to end
  Ctl* poll;           // when set: the search ends on an error or the caller's cancel word
  int wide, grow;      // wide set: the search ends at a frontier of more than wide entries,
                       // with grow also at one of more than 128 + grow * level
};

// Partition of a block's shared buffer (bytes, 16-aligned base).  vis_global:
// scratch of 2 * words words for the bitmaps when they do not fit.  Every
// thread of the block calls it.
static __device__ BlockBfs block_bfs_layout(const BlockGraph& g, unsigned char* smem, int smem_bytes,
                                            uint32_t* vis_global, int32_t* const gq[4], Ctl* poll) {
  BlockBfs b;
  b.g = g;
  b.poll = poll;
  b.wide = 0;
  b.grow = 0;
  const int words = (g.n + 31) >> 5;
  b.cnt = reinterpret_cast<int*>(smem);
  unsigned char* p = smem + 64;
  int left = smem_bytes - 64;
  const int one = (words * 4 + 15) & ~15;  // a bitmap; the slice offsets take 16 more at most
  const int qmin = 4096;                   // bytes the queues get at least
  b.sp = nullptr;
  b.dual = true;
  if (2ll * one + qmin <= left) {
    b.visA = reinterpret_cast<uint32_t*>(p);
    b.visB = reinterpret_cast<uint32_t*>(p + one);
    p += 2 * one;
    left -= 2 * one;
    if (one + 16 + qmin <= left) {
      int32_t* sp = reinterpret_cast<int32_t*>(p);
      int over = 0;
      for (int i = threadIdx.x; i <= words; i += blockDim.x) {
        sp[i] = g.slice_ptr[i];
        if (i < words && (g.slice_w[i] & kOverflowBit)) over = 1;
      }
      if (!__syncthreads_or(over)) {
        b.sp = sp;
        p += one + 16;
        left -= one + 16;
      }
    }
  } else if (one + qmin <= left) {
    b.visA = b.visB = reinterpret_cast<uint32_t*>(p);
    p += one;
    left -= one;
    b.dual = false;
  } else {
    b.visA = vis_global;
    b.visB = vis_global + words;
  }
  b.cap = left / 8;
  b.qs = reinterpret_cast<int32_t*>(p);
  b.qg0 = gq[0];
  b.qg1 = gq[1];
  b.qg2 = gq[2];
  b.qg3 = gq[3];
  return b;
}

// Entry i of the queue of a level's parity q.
static __device__ __forceinline__ int32_t* bq_at(const BlockBfs& b, int q, int i) {
  if (i < b.cap) return b.qs + q * b.cap + i;
  i -= b.cap;
  if (i < b.g.n) return (q ? b.qg2 : b.qg0) + i;
  return (q ? b.qg3 : b.qg1) + (i - b.g.n);
}

// Smallest vertex of search A in the queue of parity q (first `size`
// entries), in every thread.
static __device__ int block_queue_min(const BlockBfs& b, int q, int size) {
  if (threadIdx.x == 0) b.cnt[6] = INT_MAX;
  __syncthreads();
  int m = INT_MAX;
  for (int i = threadIdx.x; i < size; i += blockDim.x) {
    const int e = *bq_at(b, q, i);
    if (!(e & 1)) m = min(m, e >> 1);
  }
  m = __reduce_min_sync(0xffffffffu, m);
  if ((threadIdx.x & 31) == 0 && m != INT_MAX) atomicMin(&b.cnt[6], m);
  __syncthreads();
  const int r = *reinterpret_cast<volatile int*>(&b.cnt[6]);
  __syncthreads();
  return r;
}

struct BlockBfsOut {
  int la, lb;        // last non-empty level of A and of B (B: valid if !dropped)
  int t;             // smallest vertex of A's last level
  long long reached; // vertices reached by A; -1 if the search was stopped
  bool dropped;      // B was dropped because t != srcB
};

// One level: the `size` entries of the queue of parity q; claimed neighbours go
// to the other queue, their number to *cnt and B's part of it to *cntB.
// kN: neighbours a lane takes of its vertex, 8 / kN lanes a vertex.  A warp
// issues a level's instructions one after the other, and with two vertices of
// eight neighbours a lane those took most of a level (about 5,500 clocks, a
// third of it waiting for memory); a narrow frontier therefore spreads its
// neighbours over the block's lanes.  kSliced: neighbours from the sliced
// layout (b.sp), kC16: as int16 offsets; it may have been written in this
// launch, so it is read past the read-only cache.
template <bool kSliced, bool kC16, int kN>
static __device__ __forceinline__ void block_level(const BlockBfs& b, int q, int size, bool liveB, int* cnt,
                                                   int* cntB) {
  constexpr int kL = 8 / kN, kPer = 32 / kL;  // lanes a vertex, vertices a warp
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
  const int16_t* s16 = reinterpret_cast<const int16_t*>(b.g.scol);
  const int32_t* s32 = reinterpret_cast<const int32_t*>(b.g.scol);
  const int sub = (lane % kL) * kN;
  for (int base = warp * kPer; base < size; base += warps * kPer) {  // warp-uniform bound
    const int idx = base + lane / kL;
    int u = -1, e0 = 0, deg = 0, tag = 0;
    if (idx < size) {
      const int e = *bq_at(b, q, idx);
      tag = e & 1;
      if (!tag || liveB) u = e >> 1;
    }
    if (u >= 0) {
      if (kSliced) {
        const int a0 = b.sp[u >> 5], a1 = b.sp[(u >> 5) + 1];
        e0 = a0 + (u & 31);
        deg = (a1 - a0) >> 5;  // the slice's width: padding entries name the row itself
      } else {
        e0 = __ldg(&b.g.rp[u]);
        deg = __ldg(&b.g.rp[u + 1]) - e0;
      }
    }
    uint32_t* vis = tag ? b.visB : b.visA;
    const int maxdeg = __reduce_max_sync(0xffffffffu, deg);
    for (int k0 = 0; k0 < maxdeg; k0 += 8) {
      int w[kN];
#pragma unroll
      for (int j = 0; j < kN; ++j) {
        const int k = k0 + sub + j;
        w[j] = -1;
        if (k < deg) {
          if (!kSliced) w[j] = __ldg(&b.g.col[e0 + k]);
          else if (kC16) w[j] = u + (int)__ldcg(&s16[e0 + kSlice * k]);
          else w[j] = __ldcg(&s32[e0 + kSlice * k]);
        }
      }
      // the bitmap words of all candidates first, then the atomics of those
      // not visited yet
      unsigned open = 0u, push = 0u;
#pragma unroll
      for (int j = 0; j < kN; ++j)
        if (w[j] >= 0) open |= (~(*reinterpret_cast<const volatile uint32_t*>(&vis[w[j] >> 5]) >> (w[j] & 31)) & 1u) << j;
#pragma unroll
      for (int j = 0; j < kN; ++j) {
        if ((open >> j) & 1u) {
          const uint32_t bit = 1u << (w[j] & 31);
          if (!(atomicOr(&vis[w[j] >> 5], bit) & bit)) push |= 1u << j;
        }
      }
      const int m = __popc(push);
      if (!__any_sync(0xffffffffu, m)) continue;  // warp-uniform
      int inc = m;
#pragma unroll
      for (int o2 = 1; o2 < 32; o2 <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, inc, o2);
        if (lane >= o2) inc += t;
      }
      const int totB = __reduce_add_sync(0xffffffffu, tag ? m : 0);
      int at = 0;
      if (lane == 31) {
        at = atomicAdd(cnt, inc);
        if (totB) atomicAdd(cntB, totB);
      }
      int pos = __shfl_sync(0xffffffffu, at, 31) + inc - m;
#pragma unroll
      for (int j = 0; j < kN; ++j)
        if ((push >> j) & 1u) *bq_at(b, q ^ 1, pos++) = (w[j] << 1) | tag;
    }
  }
}

// Searches A from srcA and (srcB >= 0) B from srcB, level-synchronous, in
// the calling block; every thread of the block calls it.  Not inlined: the
// search then leaves the register allocation of the kernel around it alone.
template <bool kSliced, bool kC16>
static __device__ __noinline__ BlockBfsOut block_bfs2_t(const BlockBfs b, int srcA, int srcB) {
  const int tid = threadIdx.x, T = blockDim.x;
  const int words = (b.g.n + 31) >> 5;
  for (int i = tid; i < words; i += T) {
    b.visA[i] = 0u;
    b.visB[i] = 0u;
  }
  if (tid < 8) b.cnt[tid] = 0;
  __syncthreads();
  if (tid == 0) {
    b.visA[srcA >> 5] |= 1u << (srcA & 31);
    *bq_at(b, 0, 0) = srcA << 1;
    b.cnt[0] = 1;
    if (srcB >= 0) {
      b.visB[srcB >> 5] |= 1u << (srcB & 31);
      *bq_at(b, 0, 1) = (srcB << 1) | 1;
      b.cnt[0] = 2;
      b.cnt[3] = 1;
    }
  }
  __syncthreads();
  BlockBfsOut o{0, 0, -1, 0, false};
  bool liveB = srcB >= 0, doneA = false;
  int lastsize = 0;  // entries of the previous level's queue
  for (int level = 0;; ++level) {
    const int size = *reinterpret_cast<volatile int*>(&b.cnt[level % 3]);
    int sb = *reinterpret_cast<volatile int*>(&b.cnt[3 + level % 3]);
    const int sa = size - sb;
    if (sa == 0 && !doneA) {  // A has ended: its last level is known
      doneA = true;
      o.t = block_queue_min(b, (level & 1) ^ 1, lastsize);
      if (liveB && o.t != srcB) {
        liveB = false;
        o.dropped = true;
      }
    }
    if (!liveB) sb = 0;
    if (sa == 0 && sb == 0) break;
    if (b.wide && (size > b.wide || (b.grow && size > 128 + b.grow * level))) {
      o.reached = -1;
      break;
    }
    if (b.poll && (level & 255) == 255) {
      if (tid == 0 && (volatile_status(b.poll) != 0 || poll_cancel(b.poll))) b.cnt[7] = 1;
      __syncthreads();
      if (*reinterpret_cast<volatile int*>(&b.cnt[7])) {
        o.reached = -1;
        break;
      }
    }
    o.reached += sa;
    if (sa) o.la = level;
    if (sb) o.lb = level;
    lastsize = size;
    if (tid == 0) {
      b.cnt[(level + 2) % 3] = 0;
      b.cnt[3 + (level + 2) % 3] = 0;
    }
    const int q = level & 1;
    int* cnt = &b.cnt[(level + 1) % 3];
    int* cntB = &b.cnt[3 + (level + 1) % 3];
    if (8 * size <= T) block_level<kSliced, kC16, 1>(b, q, size, liveB, cnt, cntB);
    else if (4 * size <= T) block_level<kSliced, kC16, 2>(b, q, size, liveB, cnt, cntB);
    else if (2 * size <= T) block_level<kSliced, kC16, 4>(b, q, size, liveB, cnt, cntB);
    else block_level<kSliced, kC16, 8>(b, q, size, liveB, cnt, cntB);
    __syncthreads();
  }
  return o;  // unless stopped, the loop ends only after A has ended, so o.t is set
}
static __device__ BlockBfsOut block_bfs2(const BlockBfs& b, int srcA, int srcB) {
  if (!b.sp) return block_bfs2_t<false, false>(b, srcA, srcB);
  if (b.g.c16) return block_bfs2_t<true, true>(b, srcA, srcB);
  return block_bfs2_t<true, false>(b, srcA, srcB);
}

// 2BFS of a connected graph in one block.  Returns false (in every thread)
// if vertex 0 does not reach all n vertices (*apart is set) or the search was
// stopped; then nothing else is written.
static __device__ bool block_pseudo_diameter(const BlockBfs& b, int* pdiam, int* t_out, bool* apart) {
  *apart = false;
  if (b.g.n <= 0) return false;
  const int guess = b.dual ? b.g.n - 1 : -1;
  int src = 0;
  for (int pass = 0; pass < 2; ++pass) {
    const BlockBfsOut o = block_bfs2(b, src, pass == 0 ? guess : -1);
    if (o.reached != b.g.n) {
      *apart = o.reached >= 0;
      return false;
    }
    if (pass == 1) {
      *pdiam = o.la;
    } else {
      *t_out = o.t;
      if (guess >= 0 && o.t == guess && !o.dropped) {
        *pdiam = o.lb;
        break;
      }
      src = o.t;
    }
  }
  return true;
}

}  // namespace mpcg
