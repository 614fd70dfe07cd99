// cluster.cu -- the whole method (both stages) for a small system, in one
// launch of one thread-block cluster.
//
// A small system does not fill the chip: with one block per SM an iteration
// is three grid synchronisations through L2 and a chain of L2 round trips
// (measured on the 64 x 64 grid: 9.5 us a single-precision and 11.8 us a
// double-precision iteration, whatever the size up to about 60,000 rows).
// Here one cluster of 16 blocks holds the system:
//   * every block owns a contiguous range of 32-row slices and keeps them in
//     shared memory for the whole stage: values, and columns packed in 16
//     bits (owner block, row in the owner);
//   * the gathered vector d lives in the owners' shared memory and is read
//     through distributed shared memory (215 clocks against about 1,500 for a
//     write to L2, a barrier and a read back);
//   * x, r and q stay in registers: lane l of warp w owns rows
//     32 (w + 16 j) + l of its block, j < RPT, in every phase;
//   * sums go through one exchange of the 16 block partials and a hardware
//     cluster barrier (520 clocks).
// What bounds an iteration: at 4,096 rows the chain of dependent steps (FP64
// adds of the sums at 64 clocks each, one FP64 division a sum at 534 clocks,
// three cluster barriers); from about 16,000 rows the FP64 pipes of the 16
// SMs (one warp-wide FMA per 19 clocks and SM), which is why larger systems
// take the grid-wide kernels (cluster_line below).
//
// The arithmetic is that of the grid-wide kernels (cg.cu): rows summed in
// stored order by fused multiply-adds, float-float inner products in single
// precision, alpha and beta the double quotients rounded once to float.
//
// Algorithm II: the launch has two clusters.  The one that begins first runs
// the 2BFS, the other CG, whose iterations past k0 are speculative with
// snapshots at every candidate eps1, as in k_stage1.  The kNN vote is run by
// whichever comes second with its part of the features, so the 2BFS never
// waits for CG, and CG, which may wait for the label, waits for a cluster that
// has begun: the launch ends whatever the order in which its clusters are
// placed, also one after the other on a device that other work has filled.
#include <math.h>

#include "feature_block.cuh"
#include "internal.h"

namespace mpcg {

constexpr int kClThreads = 512;
constexpr int kClWarps = kClThreads / 32;
constexpr int kClSnaps = 6;       // snapshots of x~ in the workspace (as k_stage1)
constexpr int kClMaxRpt = 6;      // rows per thread of the largest instance
constexpr int kClSmem = 220 * 1024;  // dynamic shared memory a block may take

struct ClusterArgs {
  Ctl* ctl;
  const uint32_t* slice_w;
  const int32_t* slice_ptr;
  const int32_t* scol;
  const float* sv32;
  const double* sv64;
  const int32_t* rp;
  const int32_t* col;
  const double* val;
  const float* b32;
  const double* b64;
  double* x64;
  float* snap;
  int n, nslices;
  int mode;      // 0: Algorithm I, 1: Algorithm II, 2: double precision only
  int rows_cap;  // rows of the gathered vector a block has room for (the same in every block)
  int ent_cap;   // stored entries a block has room for
  BfsGraph g;    // Algorithm II
  int32_t *d1, *d2;
  KnnSpec knn;
  int smem_bytes, bfs_slot;
};

// ---------------------------------------------------------------------------------------
// Cluster primitives
// ---------------------------------------------------------------------------------------
__device__ __forceinline__ void cl_arrive() {
  asm volatile("barrier.cluster.arrive.release;" ::: "memory");
}
__device__ __forceinline__ void cl_wait() {
  asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}
__device__ __forceinline__ void cl_sync() {
  cl_arrive();
  cl_wait();
}
__device__ __forceinline__ uint32_t cl_rank() {
  uint32_t r;
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t cl_map(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void cl_ld(uint32_t addr, double& v) {
  asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(addr));
}
__device__ __forceinline__ void cl_ld(uint32_t addr, float& v) {
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(addr));
}
__device__ __forceinline__ void cl_st(uint32_t addr, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory");
}
__device__ __forceinline__ void cl_st(uint32_t addr, double v) {
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(addr), "d"(v) : "memory");
}

// Shared state of a block.  `slot` and `aux` are written by the other
// blocks; they alternate between two halves, and a half is written again
// only after every block has passed the cluster barrier of the sum between.
struct ClShared {
  double slot[2][kClBlocks];  // block partials of a sum, by rank
  double aux[2];              // word of block 0 that rides along a sum
  double part[kClThreads];
  double wpart[4];
  float ffp[2 * kClWarps];
  double val, rr;
  float fval;
  int dec, aux_i;
  int2 tab[kClWarps * kClMaxRpt];  // first entry and width | overflow flag, by slice
  int tail;                        // entries of row tails kept past the slices'
  // Algorithm II, thread 0's record of the candidate crossings (as k_stage1)
  double s_lo[17], s_hi[17], res_at[16];
  int nt[16], snap_it[kClSnaps];
  unsigned cmask, met;
};

// ---------------------------------------------------------------------------------------
// Sums over the cluster.  Every thread of every block calls them; the total
// is valid in warp 0, identical in every block.  `aux` (of block 0's thread
// 0) reaches every block's S.aux with the same barrier.
// ---------------------------------------------------------------------------------------
__device__ __forceinline__ void cl_exchange(ClShared& S, int rank, int half, double block_part,
                                            double aux) {
  const int lane = threadIdx.x & 31;
  if (threadIdx.x < 32) {
    aux = __shfl_sync(0xffffffffu, aux, 0);
    if (lane < kClBlocks) {
      cl_st(cl_map(smem_addr(&S.slot[half][rank]), lane), block_part);
      if (rank == 0) cl_st(cl_map(smem_addr(&S.aux[half]), lane), aux);
    }
  }
  cl_sync();
}

__device__ __forceinline__ double half_warp_sum(double v) {
#pragma unroll
  for (int o = kClBlocks / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Double partials: the threads' values are folded to 128 by four warps (one
// per FP64 issue port, so their adds overlap), then summed.  A dependent
// FP64 add takes 64 clocks, so 512 values summed by one warp (15 adds and a
// butterfly) took 1,430 clocks; this takes about 1,000.
__device__ __forceinline__ double cl_total(ClShared& S, int rank, int ns, int& red, double p,
                                           double aux = 0.0) {
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  const int half = red & 1;
  ++red;
  if (ns > 4) {  // otherwise only the first four warps own rows
    S.part[t] = p;
    __syncthreads();
    if (warp < 4) {
      p += S.part[t + 128];
      if (ns > 8) p += S.part[t + 256] + S.part[t + 384];
    }
  }
  if (warp < 4) {
    p = warp_sum(p);
    if (lane == 0) S.wpart[warp] = p;
  }
  __syncthreads();
  double bs = 0.0;
  if (warp == 0) bs = (S.wpart[0] + S.wpart[1]) + (S.wpart[2] + S.wpart[3]);
  cl_exchange(S, rank, half, bs, aux);
  double s = 0.0;
  if (warp == 0) s = half_warp_sum(S.slot[half][lane & (kClBlocks - 1)]);
  return s;
}

// Float-float partials.
__device__ __forceinline__ double cl_total_ff(ClShared& S, int rank, int ns, int& red, FF v,
                                              double aux = 0.0) {
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  const int half = red & 1;
  ++red;
  if (warp < ns) {
    v = ff_warp_sum(v, false);
    if (lane == 0) {
      S.ffp[2 * warp] = v.hi;
      S.ffp[2 * warp + 1] = v.lo;
    }
  }
  __syncthreads();
  double bs = 0.0;
  if (warp == 0) {
    FF w = lane < kClWarps && lane < ns ? FF{S.ffp[2 * lane], S.ffp[2 * lane + 1]} : FF{0.f, 0.f};
#pragma unroll
    for (int o = kClWarps / 2; o > 0; o >>= 1) {
      FF u;
      u.hi = __shfl_xor_sync(0xffffffffu, w.hi, o);
      u.lo = __shfl_xor_sync(0xffffffffu, w.lo, o);
      w = ff_add(w, u, false);
    }
    bs = (double)w.hi + (double)w.lo;
  }
  cl_exchange(S, rank, half, bs, aux);
  double s = 0.0;
  if (warp == 0) s = half_warp_sum(S.slot[half][lane & (kClBlocks - 1)]);
  return s;
}

// ---------------------------------------------------------------------------------------
// The system in shared memory
// ---------------------------------------------------------------------------------------
// A block's part: the gathered vector, the entries' values and packed
// columns (owner << 12 | row in the owner; rows_cap <= 3072).
//
// Where most entries lie in other blocks' rows (random graphs), a gather
// through distributed shared memory costs 52 clocks a warp (32 lanes, up to 16
// targets), and a row's gathers bound the iteration (n = 3,001 random tree:
// 4,900 of 15,500 clocks).  (8-regular graph of 2,000 rows: 6.6 us a
// double-precision iteration that way, 5.7 with whole copies; tree of 4,000
// rows 7.9 and 7.2, in single precision 7.6 and 6.1.)  Up to kClRepN rows
// every block then keeps the whole vector: the owner writes each value to all sixteen, the entries' owner is
// the block itself, and a gather stays in its own shared memory.
constexpr int kClRepN = 4096;
struct ClMat {
  unsigned char* g;   // gathered vector: rows_cap values (float or double)
  int base;           // first row of the block in g: 0, or its first row where g is whole
  bool rep;           // g is whole in every block
  unsigned char* v;   // values of the entries (float or double)
  uint16_t* c;
};

// Publish the value of one of the block's rows (`local`) in the gathered vector.
template <typename T>
__device__ __forceinline__ void cl_put(const ClMat& M, int local, T v) {
  T* g = reinterpret_cast<T*>(M.g) + M.base + local;
  if (!M.rep) {
    *g = v;
    return;
  }
  const uint32_t addr = smem_addr(g);
#pragma unroll
  for (int o = 0; o < kClBlocks; ++o) cl_st(cl_map(addr, o), v);
}

__device__ __forceinline__ uint16_t cl_pack(int nslices, int c) {
  const int o = cl_owner(nslices, c >> 5);
  return (uint16_t)((o << 12) | (c - kSlice * cl_first(nslices, o)));
}

// acc + the sum over the entries [f, f1) of one row in the caller's CSR, in
// stored order, by the whole warp (acc alike in every lane): each lane loads
// and gathers one of 32 entries, the next 32 on their way, and the chain of
// fused multiply-adds runs in every lane, so that an entry costs about its
// dependent FMA.  Stars, FP64, an iteration: 12,000 rows 0.69 ms, 2.57 by one
// lane an entry at a time and 1.08 by the grid-wide kernels; 4,000 rows 0.22,
// 0.42 and 0.37.  (Many long rows in one slice stay with their lanes: sixteen
// hubs of 20,000 rows 0.37 ms, 0.27 by the grid.)
template <typename T>
__device__ __noinline__ T cl_warp_tail(const ClusterArgs& a, bool rep, uint32_t gb, int f, int f1, T acc) {
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const uint32_t self = cl_rank() << 12;
  int c = 0;  // (a lane without an entry gathers a row that exists and is not used)
  T v = (T)0;
  if (f + lane < f1) {
    c = a.col[f + lane];
    v = (T)a.val[f + lane];
  }
  for (; f < f1; f += 32) {  // warp-uniform
    const uint32_t p = rep ? self | (uint32_t)c : (uint32_t)cl_pack(a.nslices, c);
    const T w = v;
    T x;
    cl_ld(cl_map(gb, p >> 12) + (p & 4095u) * (uint32_t)sizeof(T), x);
    if (f + 32 + lane < f1) {
      c = a.col[f + 32 + lane];
      v = (T)a.val[f + 32 + lane];
    }
    const int m = min(32, f1 - f);
    if (m == 32) {
#pragma unroll
      for (int k = 0; k < 32; ++k) acc = fma(__shfl_sync(full, w, k), __shfl_sync(full, x, k), acc);
    } else {
      for (int k = 0; k < m; ++k) acc = fma(__shfl_sync(full, w, k), __shfl_sync(full, x, k), acc);
    }
  }
  return acc;
}

// Columns once (`cols`), values at the start of each stage.  The entries of a
// row past the layout's width cap go behind the slices' where there is room
// (tail[j]: first entry | number << 16; 0: none, or read from the CSR).  Read
// from the caller's CSR at every pass, with a division for the owner of each,
// they made a random tree's SpMV three times as long as its other rows need.
// Where one or two rows of a slice have many (the hub of a star), the warp sums
// each together (kClTailWarp, whose number reads as 0).
constexpr uint32_t kClTailWarp = 0x80000000u;
constexpr int kClLongTail = 64;
template <typename T, int RPT>
__device__ __forceinline__ void cl_load(const ClusterArgs& a, ClShared& S, const ClMat& M, int S0,
                                        int rank, int ns, const T* sv, bool cols, uint32_t (&tail)[RPT]) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int E0 = a.slice_ptr[S0], E = a.slice_ptr[S0 + ns] - E0;
  const bool c16 = a.ctl->col16 != 0;
  T* vd = reinterpret_cast<T*>(M.v);
  if (cols) {
    if (threadIdx.x == 0) S.tail = 0;
    __syncthreads();
  }
#pragma unroll
  for (int j = 0; j < RPT; ++j) {
    const int s = warp + kClWarps * j;
    if (cols) tail[j] = 0u;
    if (s >= ns) continue;
    const uint32_t wf = a.slice_w[S0 + s];
    const int w = (int)(wf & ~kOverflowBit), p = a.slice_ptr[S0 + s];
    if (lane == 0) S.tab[s] = make_int2(p - E0, (int)wf);
    const int i = (S0 + s) * kSlice + lane;
    for (int k = 0; k < w; ++k) {
      const int e = p + kSlice * k + lane;
      vd[e - E0] = sv[e];
      if (cols) {
        const int c = c16 ? i + (int)reinterpret_cast<const int16_t*>(a.scol)[e] : a.scol[e];
        M.c[e - E0] = M.rep ? (uint16_t)((rank << 12) | c) : cl_pack(a.nslices, c);
      }
    }
    if (wf & kOverflowBit) {  // warp-uniform
      int e0 = 0, cnt = 0;
      if (i < a.n) {
        e0 = a.rp[i] + w;
        cnt = a.rp[i + 1] - e0;
      }
      if (cols) {
        // (rows in turn against all lanes at once: even at two rows or more)
        const unsigned lng = __ballot_sync(0xffffffffu, cnt > kClLongTail);
        if (cnt > kClLongTail && __popc(lng) <= 2) tail[j] = kClTailWarp;
      }
      if (cols && tail[j] == 0u && cnt > 0 && cnt < (1 << 15)) {
        const int at = E + atomicAdd(&S.tail, cnt);
        if (at + cnt <= a.ent_cap && at < (1 << 16)) tail[j] = (uint32_t)at | ((uint32_t)cnt << 16);
      }
      const int at = (int)(tail[j] & 0xffffu), m = (int)(tail[j] >> 16) & 0x7fff;
      for (int k = 0; k < m; ++k) {
        vd[at + k] = (T)a.val[e0 + k];
        if (cols) {
          const int c = a.col[e0 + k];
          M.c[at + k] = M.rep ? (uint16_t)((rank << 12) | c) : cl_pack(a.nslices, c);
        }
      }
    }
  }
  __syncthreads();
}

template <int RPT>
__device__ __forceinline__ bool cl_longs(const uint32_t (&tail)[RPT]) {
  uint32_t t = 0u;
#pragma unroll
  for (int j = 0; j < RPT; ++j) t |= tail[j];
  return __any_sync(0xffffffffu, (t & kClTailWarp) != 0u);
}

// acc + the sum over K entries of a row, from shared memory: all columns, then
// all gathers, then the chain of fused multiply-adds, so that a row waits once
// for its columns and once for its gathers.
template <typename T, int K>
__device__ __forceinline__ T cl_entries(uint32_t gb, const uint16_t* cp, const T* vp, T acc) {
  uint32_t c[K];
  T x[K];
#pragma unroll
  for (int k = 0; k < K; ++k) c[k] = cp[kSlice * k];
#pragma unroll
  for (int k = 0; k < K; ++k) cl_ld(cl_map(gb, c[k] >> 12) + (c[k] & 4095u) * (uint32_t)sizeof(T), x[k]);
#pragma unroll
  for (int k = 0; k < K; ++k) acc = fma(vp[kSlice * k], x[k], acc);
  return acc;
}

// Row sums of the block's slices: q[j] = sum_k v_k g(c_k) of row
// 32 (warp + 16 j) + lane, in stored order (0 where the thread has no row).
// longs (warp-uniform): some tail[j] is kClTailWarp.
template <typename T, int RPT>
__device__ __forceinline__ void cl_spmv(const ClusterArgs& a, const ClShared& S, const ClMat& M, int S0,
                                        int ns, const uint32_t (&tail)[RPT], bool longs, T (&q)[RPT]) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t gb = smem_addr(M.g);
#pragma unroll
  for (int j = 0; j < RPT; ++j) {
    const int s = warp + kClWarps * j;
    T acc = (T)0;
    if (s < ns) {
      const int2 t = S.tab[s];
      const uint32_t wf = (uint32_t)t.y;
      const int w = (int)(wf & ~kOverflowBit);
      const uint16_t* cp = M.c + t.x + lane;
      const T* vp = reinterpret_cast<const T*>(M.v) + t.x + lane;
      int k = 0;
      while (w - k > 9) {  // warp-uniform
        acc = cl_entries<T, 6>(gb, cp + kSlice * k, vp + kSlice * k, acc);
        k += 6;
      }
      cp += kSlice * k;
      vp += kSlice * k;
      switch (w - k) {
        case 1: acc = cl_entries<T, 1>(gb, cp, vp, acc); break;
        case 2: acc = cl_entries<T, 2>(gb, cp, vp, acc); break;
        case 3: acc = cl_entries<T, 3>(gb, cp, vp, acc); break;
        case 4: acc = cl_entries<T, 4>(gb, cp, vp, acc); break;
        case 5: acc = cl_entries<T, 5>(gb, cp, vp, acc); break;
        case 6: acc = cl_entries<T, 6>(gb, cp, vp, acc); break;
        case 7: acc = cl_entries<T, 7>(gb, cp, vp, acc); break;
        case 8: acc = cl_entries<T, 8>(gb, cp, vp, acc); break;
        case 9: acc = cl_entries<T, 9>(gb, cp, vp, acc); break;
        default: break;
      }
      const int i = (S0 + s) * kSlice + lane;
      if (wf & kOverflowBit) {
        const int m = (int)(tail[j] >> 16) & 0x7fff;
        const uint16_t* tc = M.c + (tail[j] & 0xffffu);
        const T* tv = reinterpret_cast<const T*>(M.v) + (tail[j] & 0xffffu);
        int e = 0;
        for (; e + 4 <= m; e += 4) {
          T x[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const uint32_t c = tc[e + u];
            cl_ld(cl_map(gb, c >> 12) + (c & 4095u) * (uint32_t)sizeof(T), x[u]);
          }
#pragma unroll
          for (int u = 0; u < 4; ++u) acc = fma(tv[e + u], x[u], acc);
        }
        for (; e < m; ++e) {
          const uint32_t c = tc[e];
          T x;
          cl_ld(cl_map(gb, c >> 12) + (c & 4095u) * (uint32_t)sizeof(T), x);
          acc = fma(tv[e], x, acc);
        }
        if (tail[j] == 0u && i < a.n) {  // no room: from the caller's CSR
          const int e1 = a.rp[i + 1];
          for (int f = a.rp[i] + w; f < e1; ++f) {
            const uint32_t c = M.rep ? (uint32_t)a.col[f] : cl_pack(a.nslices, a.col[f]);
            T x;
            cl_ld(cl_map(gb, M.rep ? cl_rank() : c >> 12) + (c & 4095u) * (uint32_t)sizeof(T), x);
            acc = fma((T)a.val[f], x, acc);
          }
        }
      }
      if (i >= a.n) acc = (T)0;
    }
    q[j] = acc;
  }
  // (in a pass of their own, which keeps the calls out of the loop above)
  if (longs) {
#pragma unroll
    for (int j = 0; j < RPT; ++j) {
      unsigned rows = __ballot_sync(0xffffffffu, tail[j] == kClTailWarp);
      while (rows) {  // warp-uniform
        const int s = warp + kClWarps * j, src = __ffs(rows) - 1, r = (S0 + s) * kSlice + src;
        rows &= rows - 1;
        const int w = (int)((uint32_t)S.tab[s].y & ~kOverflowBit);
        const T t = cl_warp_tail<T>(a, M.rep, gb, a.rp[r] + w, a.rp[r + 1], __shfl_sync(0xffffffffu, q[j], src));
        if (lane == src) q[j] = t;
      }
    }
  }
}

// ---------------------------------------------------------------------------------------
// Algorithm II: the 2BFS cluster and the vote
// ---------------------------------------------------------------------------------------
// One side of the features is complete (called by a whole warp).  The second
// of the two sides to say so runs the vote.
__device__ __forceinline__ void cl_feature_ready(const KnnSpec& knn, Ctl* ctl) {
  int second = 0;
  if ((threadIdx.x & 31) == 0) {
    __threadfence();
    second = atomicAdd(&ctl->feat_sides, 1);
    __threadfence();
  }
  if (__shfl_sync(0xffffffffu, second, 0) == 1) feature_vote(knn, ctl);
}

__device__ __noinline__ void cl_bfs(const ClusterArgs& a, unsigned char* smem) {
  const int rank = (int)cl_rank();
  const BlockGraph g{a.rp, a.col, a.slice_ptr, a.slice_w, a.scol, a.n, a.ctl->col16};
  const bool ok = feature_pdiam(g, a.g, a.d1, a.d2, smem, a.smem_bytes, a.bfs_slot,
                                (int)blockIdx.x - rank, kClBlocks);
  __syncthreads();
  if (rank == 0 && threadIdx.x < 32) {
    if (ok) cl_feature_ready(a.knn, a.ctl);
    else if (threadIdx.x == 0) atomicExch(&a.ctl->eps1_ready, -1);
  }
}

// The part of a cluster of Algorithm II, by the order in which the two begin:
// the first runs the 2BFS.
enum ClPart { kClPartNone = 0, kClPartBfs = 1, kClPartCg = 2 };
__device__ __forceinline__ double cl_part(Ctl* ctl) {
  return atomicAdd(&ctl->cl_begun, 1) == 0 ? kClPartBfs : kClPartCg;
}

// ---------------------------------------------------------------------------------------
enum ClDec { kClGo = 0, kClStop = 1, kClFail = 2, kClBroke = 3, kClLabel = 4, kClWaitLabel = 5,
             kClCap = 6 };

template <int RPT>
__global__ void __launch_bounds__(kClThreads, 1) k_cluster(ClusterArgs a) {
  extern __shared__ __align__(128) unsigned char cl_smem[];
  __shared__ ClShared S;
  Ctl* ctl = a.ctl;
  if (!ctl->small) return;
  const bool trivial = *reinterpret_cast<volatile int*>(&ctl->trivial) != 0;
  const int rank = (int)cl_rank();  // (read again where it is needed, which costs no register)
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int n = a.n;
  const int S0 = cl_first(a.nslices, rank), ns = cl_first(a.nslices, rank + 1) - S0;
  const bool lead = tid == 0, lead0 = lead && rank == 0;
  if (trivial) {  // b = 0: x = 0 solves A x = b exactly
    for (int i = S0 * kSlice + tid; i < min(n, (S0 + ns) * kSlice); i += kClThreads) a.x64[i] = 0.0;
    return;
  }
  // The blocks of the cluster leave, or take their part, together: block 0
  // decides for all (the other cluster may set the status at any time).  The
  // first barrier makes sure that every block runs before its memory is
  // written to.
  cl_sync();
  int red = 1;
  double part = kClPartCg;
  if (lead0) part = volatile_status(ctl) != 0 ? kClPartNone : a.mode == 1 ? cl_part(ctl) : kClPartCg;
  cl_exchange(S, rank, 0, 0.0, part);
  part = S.aux[0];
  if (part != kClPartCg) {
    if (part == kClPartBfs) cl_bfs(a, cl_smem);
    return;
  }
  ClMat M;
  M.g = cl_smem;
  M.v = M.g + (size_t)a.rows_cap * sizeof(double);
  M.c = reinterpret_cast<uint16_t*>(M.v + (size_t)a.ent_cap * sizeof(double));
  M.rep = false;
  if (n <= kClRepN) {  // uniform: count the entries in other blocks' rows
    const int E0 = a.slice_ptr[S0], E1 = a.slice_ptr[S0 + ns];
    const bool c16 = ctl->col16 != 0;
    int far = 0;
    for (int s = warp; s < ns; s += kClWarps) {
      const int w = (int)(a.slice_w[S0 + s] & ~kOverflowBit), p = a.slice_ptr[S0 + s];
      const int i = (S0 + s) * kSlice + lane;
      for (int k = 0; k < w; ++k) {
        const int e = p + kSlice * k + lane;
        const int c = c16 ? i + (int)reinterpret_cast<const int16_t*>(a.scol)[e] : a.scol[e];
        if (c < S0 * kSlice || c >= (S0 + ns) * kSlice) ++far;
      }
    }
    if (tid == 0) S.tail = 0;
    __syncthreads();
    far = __reduce_add_sync(0xffffffffu, far);
    if (lane == 0 && far) atomicAdd(&S.tail, far);
    __syncthreads();
    const int half = red & 1;
    ++red;
    cl_exchange(S, rank, half, (double)(3 * S.tail - (E1 - E0)), 0.0);
    double sum = 0.0;
    for (int o = 0; o < kClBlocks; ++o) sum += S.slot[half][o];  // exact: small whole numbers
    M.rep = sum > 0.0;  // more than a third of the stored entries (padding included)
  }
  M.base = M.rep ? S0 * kSlice : 0;
  const int rel = ctl->tol_relative;
  bool ok = true;
  int row[RPT];  // the thread's rows, or -1
#pragma unroll
  for (int j = 0; j < RPT; ++j) {
    const int s = warp + kClWarps * j, i = (S0 + s) * kSlice + lane;
    row[j] = s < ns && i < n ? i : -1;
  }
  uint32_t tail[RPT];  // where the entries past the width cap are (cl_load)
  double xd[RPT];
#pragma unroll
  for (int j = 0; j < RPT; ++j) xd[j] = 0.0;

  // =================== single-precision stage ===================
  if (a.mode != 2) {
    cl_load<float, RPT>(a, S, M, S0, rank, ns, a.sv32, true, tail);
    const bool longs = cl_longs<RPT>(tail);
    const float* g = reinterpret_cast<const float*>(M.g) + M.base;
    const bool autom = a.mode == 1;
    const int max1 = ctl->max1, k0 = ctl->k0;
    const double eps2 = ctl->eps2;
    float x[RPT], r[RPT], q[RPT];
    if (autom) {  // classes present in the sample
      if (lead) {
        S.cmask = 0u;
        S.met = 0u;
      }
      __syncthreads();
      unsigned cm = 0u;
      for (int i = tid; i < a.knn.count; i += kClThreads) {
        const int c = a.knn.cls[i];
        if (c >= 0 && c < 16) cm |= 1u << c;
      }
      cm = __reduce_or_sync(0xffffffffu, cm);
      if (lane == 0 && cm) atomicOr(&S.cmask, cm);
    }
    // CG line 1: x0 = 0, r0 = b~, d0 = r0
    FF acc{0.f, 0.f};
#pragma unroll
    for (int j = 0; j < RPT; ++j) {
      x[j] = 0.0f;
      r[j] = row[j] >= 0 ? a.b32[row[j]] : 0.0f;
      if (warp + kClWarps * j < ns) cl_put(M, (warp + kClWarps * j) * kSlice + lane, r[j]);
      if (row[j] >= 0) ff_add_prod(acc, r[j], r[j], false);
    }
    double rr = cl_total_ff(S, rank, ns, red, acc);  // the barrier also publishes d
    double bnorm = 0.0;
    if (warp == 0) {
      bnorm = sqrt(rr);
      if (lead) S.val = bnorm;
      if (lead0) {
        ctl->bnorm32 = bnorm;
        if (!isfinite(bnorm)) set_status(ctl, MPCG_ERR_NAN);
      }
    }
    __syncthreads();
    bnorm = S.val;
    if (!isfinite(bnorm)) ok = false;
    // warp 0 (all lanes alike): the state of the iteration
    int it = 0, k0done = 0, in_k0 = autom ? 1 : 0, cls = -1, nslots = 0, broke = 0;
    double vsum = 0.0;
    const StopThr thr = stop_thr(autom ? eps2 : ctl->eps1, bnorm, rel);
    if (autom && lead) {
      for (int t = 0; t < 16; ++t) {
        const StopThr c = stop_thr(pow10_neg(t), bnorm, rel);
        S.s_lo[t] = c.lo;
        S.s_hi[t] = c.hi;
        S.nt[t] = -1;
        S.res_at[t] = 0.0;
      }
    }
    __syncwarp();
    bool cancelled = false, by_label = false;
    while (ok) {
      // ---- loop head (warp 0): the stop test, and Algorithm II's record ----
      if (warp == 0) {
        int dec = kClGo, snap_slot = -1;
        if (cancelled) {
          dec = kClFail;
          if (lead0) set_status(ctl, MPCG_ERR_CANCELLED);
        } else if (bits_nan(rr)) {
          dec = kClFail;
          if (lead0) set_status(ctl, MPCG_ERR_NAN);
        } else if (!autom) {
          if (stop_pass(thr, rr) || it >= max1) dec = kClStop;
        } else {
          if (in_k0 && (it >= min(k0, max1) || dbits(rr) == 0 || stop_pass(thr, rr))) {
            in_k0 = 0;  // end of the k0 phase: v of Eq. (13)
            if (rank == 0) {
              if (lane == 0) {
                ctl->k0_done = k0done;
                ctl->vsum = vsum;
                ctl->v = k0done > 0 ? vsum / (double)k0done : 0.0;
              }
              cl_feature_ready(a.knn, ctl);
            }
          }
          if (!in_k0) {
            // Candidates are met in the order of t: above the upper bracket of
            // the lowest present class not met yet, none is met now.
            bool fresh = false;
            const unsigned open = S.cmask & ~S.met;
            __syncwarp();
            if (open && dbits(rr) <= dbits(S.s_hi[__ffs(open) - 1])) {
              unsigned met = S.met;
              __syncwarp();
              for (int t = 0; t < 16; ++t) {
                if (!((open >> t) & 1u)) continue;
                if (rr <= S.s_lo[t] || (rr <= S.s_hi[t] && stop_measure(rr, bnorm, rel) <= pow10_neg(t))) {
                  if (lane == 0) {
                    S.nt[t] = it;
                    S.res_at[t] = stop_measure(rr, bnorm, rel);
                  }
                  met |= 1u << t;
                  fresh = true;
                }
              }
              if (lane == 0) S.met = met;
              __syncwarp();
            }
            const bool all = (S.cmask & ~S.met) == 0u;
            if (cls < 0 && (all || it >= max1)) {
              dec = kClLabel;  // stage 1 ends here whatever the label
            } else if (cls < 0 && fresh && nslots >= kClSnaps) {
              dec = kClWaitLabel;
            } else if (cls < 0) {
              if (fresh) {
                snap_slot = nslots;
                if (lane == 0) S.snap_it[nslots] = it;
                ++nslots;
              }
            } else if (S.nt[cls] >= 0 || it >= max1) {
              dec = kClStop;
            }
          }
        }
        if (lane == 0) {
          S.dec = dec;
          S.aux_i = snap_slot;
        }
      }
      __syncthreads();
      int dec = S.dec;
      const int snap_slot = S.aux_i;
      if (snap_slot >= 0) {
        float* dst = a.snap + (size_t)snap_slot * n;
#pragma unroll
        for (int j = 0; j < RPT; ++j)
          if (row[j] >= 0) dst[row[j]] = x[j];
      }
      if (dec == kClWaitLabel) {  // no snapshot left: block 0 waits (bounded) and tells the others
        double lab = 0.0;
        if (rank == 0 && warp == 0) {
          int l = 0;
          if (lane == 0) l = wait_label(ctl);
          lab = (double)__shfl_sync(0xffffffffu, l, 0);
        }
        const int half = red & 1;
        ++red;
        cl_exchange(S, rank, half, 0.0, lab);
        const int l = (int)S.aux[half];
        if (warp == 0) cls = l;
        dec = l < 0 ? kClFail : (S.nt[l] >= 0 || it >= max1 ? kClStop : kClGo);
      }
      if (dec == kClLabel) by_label = true;
      if (dec == kClFail) ok = false;
      if (dec != kClGo) break;

      // ---- q = A d, d^T q ----
      int cw = 0, label_now = 0;
      if (lead0) {  // read now, used with the r^T r sum: their latency overlaps the iteration
        cw = cancel_word(ctl);
        if (autom && cls < 0) label_now = *reinterpret_cast<volatile int*>(&ctl->eps1_ready);
      }
      cl_spmv<float, RPT>(a, S, M, S0, ns, tail, longs, q);
      FF pdq{0.f, 0.f};
      float d[RPT];
#pragma unroll
      for (int j = 0; j < RPT; ++j) {
        d[j] = 0.0f;
        if (row[j] >= 0) {
          d[j] = g[row[j] - S0 * kSlice];
          ff_add_prod(pdq, d[j], q[j], false);
        }
      }
      const double dq = cl_total_ff(S, rank, ns, red, pdq);
      if (warp == 0) {
        int d2 = kClGo;
        if (!bits_finite(dq)) {
          d2 = kClFail;
          if (lead0) set_status(ctl, MPCG_ERR_NAN);
        } else if (!bits_positive(dq)) {
          d2 = kClBroke;  // stage 1 ends here; x~ and r are unchanged
        } else if (lane == 0) {
          S.fval = (float)(rr / dq);
        }
        if (lane == 0) S.dec = d2;
      }
      __syncthreads();
      dec = S.dec;
      if (dec == kClFail) ok = false;
      if (dec == kClBroke) broke = 1;
      if (dec != kClGo) break;
      const float alpha = S.fval;

      // ---- x += alpha d, r -= alpha q, r^T r ----
      FF prr{0.f, 0.f};
#pragma unroll
      for (int j = 0; j < RPT; ++j) {
        x[j] = __fmaf_rn(alpha, d[j], x[j]);
        r[j] = __fmaf_rn(-alpha, q[j], r[j]);
        if (row[j] >= 0) ff_add_prod(prr, r[j], r[j], false);
      }
      // block 0's word: 100 = cancelled, else the label (0 unknown, t + 1, or -1)
      const int half = red & 1;
      const double rrn = cl_total_ff(S, rank, ns, red, prr, (double)(cw != 0 ? 100 : label_now));
      if (warp == 0) {
        int d3 = kClGo;
        const int word = (int)S.aux[half];
        cancelled = word == 100;
        if (word < 0) {
          d3 = kClFail;
        } else if (!bits_finite(rrn)) {
          d3 = kClFail;
          if (lead0) set_status(ctl, MPCG_ERR_NAN);
        } else {
          if (!cancelled && word > 0) cls = word - 1;
          if (in_k0) {
            vsum += sqrt(rrn) / sqrt(rr);  // Eq. (13) ratio
            ++k0done;
          }
          if (lane == 0) S.fval = (float)(rrn / rr);
          rr = rrn;
        }
        if (lane == 0) S.dec = d3;
      }
      __syncthreads();
      if (S.dec != kClGo) {
        ok = false;
        break;
      }
      const float beta = S.fval;
      // ---- d = r + beta d ----
#pragma unroll
      for (int j = 0; j < RPT; ++j)
        if (row[j] >= 0) cl_put(M, row[j] - S0 * kSlice, __fmaf_rn(beta, d[j], r[j]));
      ++it;
      cl_sync();
    }
    // ---- end of the stage ----
    __syncthreads();  // every thread has read the last decision
    if (autom && ok) {
      if (warp == 0 && rank == 0 && broke && in_k0) {  // breakdown in the k0 phase
        if (lane == 0) {
          ctl->k0_done = k0done;
          ctl->vsum = vsum;
          ctl->v = k0done > 0 ? vsum / (double)k0done : 0.0;
        }
        cl_feature_ready(a.knn, ctl);
      }
      if (by_label || broke) {  // uniform: block 0 waits (bounded) and tells the others
        double lab = 0.0;
        if (rank == 0 && warp == 0) {
          int l = cls;
          if (lane == 0 && cls < 0) l = wait_label(ctl);
          lab = (double)__shfl_sync(0xffffffffu, l, 0);
        }
        const int half = red & 1;
        ++red;
        cl_exchange(S, rank, half, 0.0, lab);
        if (warp == 0) cls = (int)S.aux[half];
      }
    }
    if (warp == 0) {
      int src = -1, good = ok ? 1 : 0;
      if (ok) {
        int n1 = it;
        double res = stop_measure(rr, bnorm, rel), eps1 = autom ? 0.0 : ctl->eps1;
        if (autom) {
          if (cls < 0) {
            good = 0;
          } else {
            // the first iteration >= k0 that met eps1 = 10^-t, with its iterate;
            // otherwise (cap, breakdown) the current one
            eps1 = pow10_neg(cls);
            if (!in_k0 && S.nt[cls] >= 0 && S.nt[cls] < it) {
              n1 = S.nt[cls];
              res = S.res_at[cls];
              for (int k = 0; k < nslots; ++k)
                if (S.snap_it[k] == n1) src = k;
            }
          }
        }
        if (lead0 && good) {
          ctl->n1 = n1;
          ctl->x32_src = src;
          ctl->res32 = res;
          ctl->rr = rr;
          if (broke) ctl->broke32 = 1;
          if (res > eps1) ctl->warn_eps1 = 1;
          ctl->t_fp32 = globaltimer();
        }
      }
      if (lane == 0) {
        S.dec = good;
        S.aux_i = src;
      }
    }
    __syncthreads();
    if (!S.dec) {  // an error (its status is set), the same in every block
      cl_sync();   // no block leaves while another may still write to it
      return;
    }
    const int src = S.aux_i;
#pragma unroll
    for (int j = 0; j < RPT; ++j) {
      if (row[j] >= 0) xd[j] = (double)(src >= 0 ? a.snap[(size_t)src * n + row[j]] : x[j]);
    }
    __syncthreads();
  }

  // =================== double-precision stage ===================
  cl_load<double, RPT>(a, S, M, S0, rank, ns, a.sv64, a.mode == 2, tail);
  const bool longs = cl_longs<RPT>(tail);
  const double* g = reinterpret_cast<const double*>(M.g) + M.base;
  const double bnorm = ctl->bnorm64, eps2 = ctl->eps2;
  const int max2 = ctl->max2, max_restarts = ctl->max_restarts;
  const StopThr thr2 = stop_thr(eps2, bnorm, rel);
  double r[RPT], q[RPT];
  int it = 0, restarts = 0, failed = 0;
  double rr = 0.0, true_rel = NAN;
  int leg = 0;  // the residual pass: 0 = first, 1 = at convergence, 2 = after the cap
  for (;;) {
    // ---- residual pass: t = b - A x, ||t||^2 ----
    cl_sync();  // every block has read d (and loaded its entries)
#pragma unroll
    for (int j = 0; j < RPT; ++j)
      if (warp + kClWarps * j < ns) cl_put(M, (warp + kClWarps * j) * kSlice + lane, xd[j]);
    cl_sync();
    cl_spmv<double, RPT>(a, S, M, S0, ns, tail, longs, q);
    double p = 0.0;
#pragma unroll
    for (int j = 0; j < RPT; ++j) {
      if (warp + kClWarps * j < ns) {
        __syncwarp();
        q[j] = row[j] >= 0 ? a.b64[row[j]] - q[j] : 0.0;
        p = __fma_rn(q[j], q[j], p);
      }
    }
    int cw = lead0 ? cancel_word(ctl) : 0;
    int half = red & 1;
    const double tot = cl_total(S, rank, ns, red, p, (double)cw);
    // loop head: the stop test on the recursive residual
    auto head = [&](double rrv, int itv, bool cancelled) -> int {
      if (cancelled) {
        failed = MPCG_ERR_CANCELLED;
        return kClFail;
      }
      if (bits_nan(rrv)) {
        failed = MPCG_ERR_NAN;
        return kClFail;
      }
      if (stop_pass(thr2, rrv)) return kClStop;
      if (itv >= max2) return kClCap;
      return kClGo;
    };
    if (warp == 0) {
      int dec = kClGo;
      if (leg != 0) {
        true_rel = bnorm > 0.0 ? sqrt(tot) / bnorm : sqrt(tot);
        const double tm = rel ? true_rel : sqrt(tot);
        dec = kClFail;  // ends here
        if (leg == 1 && tm > eps2) {
          if (restarts < max_restarts) {
            ++restarts;
            dec = kClGo;
          } else {
            failed = MPCG_ERR_NOT_CONVERGED;  // the last restart still missed eps2
          }
        }
      }
      if (dec == kClGo) {
        rr = tot;
        dec = head(rr, it, dbits(S.aux[half]) != 0);
      }
      if (lane == 0) S.dec = dec;
    }
    __syncthreads();
    int dec = S.dec;
    if (dec == kClFail) break;
    if (dec == kClGo) {
#pragma unroll
      for (int j = 0; j < RPT; ++j) {
        r[j] = q[j];
        if (warp + kClWarps * j < ns) cl_put(M, (warp + kClWarps * j) * kSlice + lane, r[j]);
      }
      cl_sync();
    }
    while (dec == kClGo) {
      if (lead0) cw = cancel_word(ctl);  // used with the r^T r sum
      // ---- q = A d, d^T q ----
      cl_spmv<double, RPT>(a, S, M, S0, ns, tail, longs, q);
      // (A predicated-off FP64 instruction takes its turn of the FP64 pipe:
      // warps without a slice branch around these.  The __syncwarp keeps the
      // compiler from predicating the short bodies.)
      double pq = 0.0, d[RPT];
#pragma unroll
      for (int j = 0; j < RPT; ++j) {
        d[j] = 0.0;
        if (warp + kClWarps * j < ns) {
          __syncwarp();
          d[j] = g[(warp + kClWarps * j) * kSlice + lane];
          pq = __fma_rn(d[j], q[j], pq);
        }
      }
      const double dq = cl_total(S, rank, ns, red, pq);
      if (warp == 0) {
        int d2 = kClGo;
        if (!bits_finite(dq)) failed = MPCG_ERR_NAN;
        else if (!bits_positive(dq)) failed = MPCG_ERR_BREAKDOWN;
        else if (lane == 0) S.val = rr / dq;
        if (failed) d2 = kClFail;
        if (lane == 0) S.dec = d2;
      }
      __syncthreads();
      dec = S.dec;
      if (dec != kClGo) break;
      const double alpha = S.val;
      // ---- r -= alpha q, r^T r ----
      double pr = 0.0;
#pragma unroll
      for (int j = 0; j < RPT; ++j) {
        if (warp + kClWarps * j < ns) {
          __syncwarp();
          r[j] = __fma_rn(-alpha, q[j], r[j]);
          pr = __fma_rn(r[j], r[j], pr);
        }
      }
      half = red & 1;
      const double rrn = cl_total(S, rank, ns, red, pr, (double)cw);
      if (warp == 0) {
        int d3 = kClFail;
        if (!bits_finite(rrn)) {
          failed = MPCG_ERR_NAN;
          if (lane == 0) S.aux_i = 0;  // x keeps the iterate before the failing step
        } else {
          d3 = head(rrn, it + 1, dbits(S.aux[half]) != 0);
          if (lane == 0) {
            S.val = rrn / rr;  // beta
            S.aux_i = 1;
          }
          rr = rrn;
        }
        if (lane == 0) S.dec = d3;
      }
      __syncthreads();
      dec = S.dec;
      const int step = S.aux_i;
      const double beta = S.val;
      if (!step) break;
      // ---- d = r + beta d, x += alpha d ----
      if (dec == kClGo) {
#pragma unroll
        for (int j = 0; j < RPT; ++j) {
          if (warp + kClWarps * j < ns) {
            __syncwarp();
            cl_put(M, (warp + kClWarps * j) * kSlice + lane, __fma_rn(beta, d[j], r[j]));
          }
        }
        cl_arrive();
      }
#pragma unroll
      for (int j = 0; j < RPT; ++j) {
        if (warp + kClWarps * j < ns) {
          __syncwarp();
          xd[j] = __fma_rn(alpha, d[j], xd[j]);
        }
      }
      ++it;
      if (dec == kClGo) cl_wait();
    }
    if (dec == kClFail) break;
    leg = dec == kClStop ? 1 : 2;
    if (leg == 2) failed = MPCG_ERR_NOT_CONVERGED;
  }
#pragma unroll
  for (int j = 0; j < RPT; ++j)
    if (row[j] >= 0) a.x64[row[j]] = xd[j];
  if (lead0) {
    if (failed) set_status(ctl, failed);
    ctl->n2 = it;
    ctl->restarts = restarts;
    if (restarts) ctl->warn_restart = 1;
    ctl->res64 = stop_measure(rr, bnorm, rel);
    ctl->true_rel = true_rel;
    ctl->rr = rr;
    ctl->t_fp64 = globaltimer();
  }
  cl_sync();  // no block leaves while another may still read or write its shared memory
}

// ---------------------------------------------------------------------------------------
// Host
// ---------------------------------------------------------------------------------------
namespace {

const void* cluster_kernel(int rpt) {
  switch (rpt) {
    case 1: return (const void*)k_cluster<1>;
    case 2: return (const void*)k_cluster<2>;
    case 4: return (const void*)k_cluster<4>;
    default: return (const void*)k_cluster<kClMaxRpt>;
  }
}

// Rows per thread of the instance for n rows; 0: none is large enough.
int cluster_rpt(int nslices) {
  const int per_block = (nslices + kClBlocks - 1) / kClBlocks;
  const int rpt = (per_block + kClWarps - 1) / kClWarps;
  return rpt <= 1 ? 1 : rpt <= 2 ? 2 : rpt <= 4 ? 4 : rpt <= kClMaxRpt ? kClMaxRpt : 0;
}

size_t cluster_smem(const Dims& d, int* rows_cap, int* ent_cap) {
  const int rows = (d.nslices + kClBlocks - 1) / kClBlocks * kSlice;
  *rows_cap = d.n <= kClRepN ? d.nslices * kSlice : rows;
  *ent_cap = rows * d.wcap;
  return (size_t)*rows_cap * sizeof(double) + (size_t)*ent_cap * (sizeof(double) + sizeof(uint16_t));
}

// Whether the device takes a cluster of kClBlocks blocks of every instance
// (and the attributes that such launches need are set).  Per device; a benign
// race between host threads computes the same value twice.
bool cluster_device_ok() {
  constexpr int kMaxDevices = 64;
  static int cached[kMaxDevices];  // 0 unknown, 1 yes, -1 no
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return false;
  if (!cached[dev]) {
    int good = 1;
    for (int rpt : {1, 2, 4, kClMaxRpt}) {
      const void* k = cluster_kernel(rpt);
      if (cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
          cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kClSmem) != cudaSuccess) {
        good = -1;
        break;
      }
      cudaLaunchConfig_t cfg = {};
      cudaLaunchAttribute at[1];
      at[0].id = cudaLaunchAttributeClusterDimension;
      at[0].val.clusterDim.x = kClBlocks;
      at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
      cfg.gridDim = dim3(kClBlocks);
      cfg.blockDim = dim3(kClThreads);
      cfg.dynamicSmemBytes = kClSmem;
      cfg.attrs = at;
      cfg.numAttrs = 1;
      int clusters = 0;
      if (cudaOccupancyMaxActiveClusters(&clusters, k, &cfg) != cudaSuccess || clusters < 1) {
        good = -1;
        break;
      }
    }
    if (good < 0) (void)cudaGetLastError();  // a refused attribute is no error of the call
    cached[dev] = good;
  }
  return cached[dev] > 0;
}

}  // namespace

// The line between the cluster and the grid-wide kernels: the block's part
// fits in shared memory for every sparsity pattern with these counts, and
// nnz + 5 n, the FP64 FMAs of an iteration, is at most kClMaxFma.
//
// Past kClRepN rows, where d is read from its owners, the gathers of a matrix
// whose columns are scattered bound the iteration: 52 clocks for one whose
// lanes reach most of the blocks.  The host does not know the pattern, so the
// set-up counts the entries in other blocks' rows whose gather reaches four
// blocks or more, and the cluster takes at most kClMaxFar of them.  Where the
// two ways are even (FP64 solves): 8-regular graphs at 6,100 rows (46,000 such
// entries; 0.43 ms), 4-regular at 12,500 (47,000; 0.60 ms), trees with n / 2
// more edges at 16,000 (44,000; 11.6 ms), trees at 28,500 (52,000; 26 ms).
// Past it (us, cluster and grid): 8-regular graph of 20,000 rows 861 and 458,
// tree with n / 2 more edges of 36,000 rows 33,600 and 22,100.  Stencils and
// bands have no such entries (a gather reaches two blocks, or three).
//
// The kernels not taken leave at once, 6 us each (3 % of the shortest solve, a
// band of width 15 and 6,000 rows), so they are not launched where the
// entries off the diagonal, of which a scattered matrix has fifteen of sixteen
// in other blocks, keep the count below the line (kClMaxOff).
constexpr long long kClMaxFma = 400000;
constexpr int kClMaxFar = 45000;
constexpr int kClMaxOff = 48000;

int cluster_line(const Dims& d) {
  int rows, ents;
  const bool fits = cluster_rpt(d.nslices) > 0 && (long long)d.nnz + 5ll * d.n <= kClMaxFma &&
                    cluster_smem(d, &rows, &ents) <= (size_t)kClSmem && cluster_device_ok();
  if (!fits) return -1;
  return d.n <= kClRepN || d.nnz - d.n <= kClMaxOff ? kClAlways : kClMaxFar;
}

cudaError_t launch_cluster(const Launch& L, const double* b, double* x, const mpcg_sample_t* S,
                           const mpcg_options_t& o, int mode, int bfs_slot) {
  ClusterArgs a{};
  a.bfs_slot = bfs_slot;
  a.ctl = L.ws.ctl;
  a.slice_w = L.ws.slice_w;
  a.slice_ptr = L.ws.slice_ptr;
  a.scol = L.ws.scol;
  a.sv32 = L.ws.sv32;
  a.sv64 = L.ws.sv64;
  a.rp = L.A->row_ptr;
  a.col = L.A->col;
  a.val = L.A->val;
  a.b32 = L.ws.b32;
  a.b64 = b;
  a.x64 = x;
  a.snap = L.ws.snap;
  a.n = L.d.n;
  a.nslices = L.d.nslices;
  a.mode = mode;
  a.g = bfs_graph(L);
  a.d1 = L.ws.dist;
  a.d2 = L.ws.dist2;
  if (mode == 1) a.knn = knn_spec(*S, o);
  size_t smem = cluster_smem(L.d, &a.rows_cap, &a.ent_cap);
  if (mode == 1) smem = kClSmem;  // the 2BFS's bitmaps and queues
  a.smem_bytes = (int)smem;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = kClBlocks;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.gridDim = dim3(mode == 1 ? 2 * kClBlocks : kClBlocks);
  cfg.blockDim = dim3(kClThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = L.st;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  void* args[] = {&a};
  return cudaLaunchKernelExC(&cfg, cluster_kernel(cluster_rpt(L.d.nslices)), args);
}

}  // namespace mpcg
