// feature_block.cuh -- the features of Algorithm II by one block beside the
// blocks that run CG (the cluster kernel and the fused single-precision stage).
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

// The block's own barrier as the group barrier of the 2BFS routines.
struct BlockSync {
  static constexpr bool kWholeBlock = true;
  static constexpr bool kNarrow = false;
  static constexpr bool kHelpers = false;
  Ctl* ctl;
  __device__ bool operator()() {
    __shared__ int s_ok;
    __syncthreads();
    if (threadIdx.x == 0) s_ok = volatile_status(ctl) == 0 && !poll_cancel(ctl);
    __syncthreads();
    return s_ok != 0;
  }
};

// l~ by the calling block, into the control block: the one-block search, or,
// where the graph has more than one component, the group's routines over this
// block.  False (in every thread) on an error or a cancel.
static __device__ bool block_pdiam_any(Ctl* ctl, const int32_t* rp, const int32_t* col, const int32_t* slice_ptr,
                                       const uint32_t* slice_w, const void* scol, int n, const BfsGraph& q,
                                       int32_t* d1, int32_t* d2, unsigned char* smem, int smem_bytes) {
  int32_t* const gq[4] = {q.fq0, q.fq1, q.fq2, q.fq3};
  const BlockGraph g{rp, col, slice_ptr, slice_w, scol, n, ctl->col16};
  const BlockBfs b = block_bfs_layout(g, smem, smem_bytes, reinterpret_cast<uint32_t*>(q.ckey), gq, ctl);
  int pd = 0, tv = 0;
  bool ok = block_pseudo_diameter(b, &pd, &tv);
  __syncthreads();
  if (ok) {
    if (threadIdx.x == 0) {
      ctl->pdiam = pd;
      ctl->far_t = tv;
      ctl->reached = n;
      ctl->connected = 1;
    }
  } else {  // more than one component (or an error, which the group barrier reports)
    BlockSync sync{ctl};
    ok = pseudo_diameter_run<BlockSync, false>(q, d1, d2, threadIdx.x, blockDim.x, sync);
  }
  return ok;
}

}  // namespace mpcg
