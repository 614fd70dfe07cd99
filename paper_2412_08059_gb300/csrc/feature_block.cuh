// feature_block.cuh -- the features of Algorithm II by one block, or by a
// group of blocks beside those that run CG (the cluster kernel and the fused
// single-precision stage).
#pragma once
#include "bfs_block.cuh"
#include "bfs_core.cuh"
#include "knn_core.cuh"

namespace mpcg {

// The vote from the features in the control block, by one warp; publishes
// the label (or the failure).
static __device__ __noinline__ void feature_vote(const KnnSpec& knn, Ctl* ctl) {
  const volatile Ctl* c = ctl;
  const double chi[4] = {(double)c->n, (double)c->nnz, (double)c->pdiam, c->v};
  const int t = knn_warp(knn, chi);
  if ((threadIdx.x & 31) == 0) {
    if (t >= 0) {
      ctl->cls = t;
      ctl->eps1 = pow10_neg(t);
    } else {
      set_status(ctl, MPCG_ERR_INVALID_ARG);  // invalid query, sample or label
    }
    ctl->t_features = globaltimer();
    __threadfence();
    atomicExch(&ctl->eps1_ready, t >= 0 ? t + 1 : -1);
  }
  __syncwarp();
}

// Sizes the one-block search takes (bfs_block.cuh) before the blocks of a
// group, or of the grid, search together, and the frontiers at which it gives
// up for them (entries of both searches).  Up to kPdSmallN vertices 2,048: a
// whole cube is then no slower than by the grid (features of 24^3: 0.58 ms
// against 0.67; of 32^3 0.95 against 0.84).  Past it 128 + 8 level, at most
// 1,280: a 2-D grid (2 level) of up to kPdMaxN vertices stays within that (512 x
// 512: 5.5 against 5.9 ms), a cube leaves it at level 16 (level^2), some 50 us
// into a search of a millisecond.  A larger square grid would leave it late
// (700 x 700: 12.8 ms against 8.8), so larger graphs are not tried; that the
// line is drawn by n keeps long thin grids past it, which would stay within
// the limits, with the search of all blocks (5 to 6 us a level).
constexpr int kPdMaxN = 300000;
constexpr int kPdSmallN = 16384;

// l~ by the calling block, into the control block (pd_done set).  False (in
// every thread) if the graph has more than one component (pd_apart set: the
// group goes on with the components, without another search from vertex 0),
// its frontier grows past the limits, or on an error or a cancel.
static __device__ bool block_pdiam(const BlockGraph& g, const BfsGraph& q, unsigned char* smem, int smem_bytes) {
  Ctl* ctl = q.ctl;
  int32_t* const gq[4] = {q.fq0, q.fq1, q.fq2, q.fq3};
  BlockBfs b = block_bfs_layout(g, smem, smem_bytes, reinterpret_cast<uint32_t*>(q.ckey), gq, ctl);
  b.wide = g.n <= kPdSmallN ? 2048 : 1280;
  b.grow = g.n <= kPdSmallN ? 0 : 8;
  int pd = 0, tv = 0;
  bool apart = false;
  const bool ok = block_pseudo_diameter(b, &pd, &tv, &apart);
  __syncthreads();
  if (apart && threadIdx.x == 0) ctl->pd_apart = 1;
  if (ok && threadIdx.x == 0) {
    ctl->pdiam = pd;
    ctl->far_t = tv;
    ctl->reached = g.n;
    ctl->connected = 1;
    ctl->pd_done = 1;
  }
  return ok;
}

// l~ by a group of blocks of a launch that run beside the CG blocks: `blocks`
// of them from `first` on.  The first tries the one-block search while the
// others wait at the group's (bounded) barrier; where it gives up, they search
// together.  False (in every thread) on an error or a cancel.
static __device__ bool feature_pdiam(const BlockGraph& g, const BfsGraph& q, int32_t* d1, int32_t* d2,
                                     unsigned char* smem, int smem_bytes, int slot, int first, int blocks) {
  const int rank = (int)blockIdx.x - first;
  if (rank == 0 && g.n <= kPdMaxN) block_pdiam(g, q, smem, smem_bytes);
  BlockGroupSync sync{q.ctl, slot, 0ull, blocks, reinterpret_cast<int*>(smem)};
  if (!sync()) return false;
  if (*reinterpret_cast<volatile int*>(&q.ctl->pd_done)) return true;
  return pseudo_diameter_run<BlockGroupSync, false>(q, d1, d2, rank * (int)blockDim.x + (int)threadIdx.x,
                                                    blocks * (int)blockDim.x, sync);
}

}  // namespace mpcg
