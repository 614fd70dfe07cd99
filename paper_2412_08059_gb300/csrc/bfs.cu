// bfs.cu -- standalone kernels for the sparsity-graph features of Sec. 6
// (the routines are in bfs_core.cuh and bfs_block.cuh): the 2BFS
// pseudo-diameter, with the per-component rule, by one block or in one
// cooperative launch, and a plain BFS.
#include "feature_block.cuh"
#include "internal.h"

namespace mpcg {

// The 2BFS by one block (bfs_block.cuh).  A level costs the grid-wide search
// its barriers and a chain of L2 round trips, 5 to 6 us whatever its width up
// to a few thousand vertices; here 2.7 us at 128 entries (both searches
// together) and 5.3 us at 1,000, so long thin graphs gain most (4096 x 64
// grid, 4,158 levels: 21.7 ms by the grid, 11.4 here).  A frontier that grows
// like a cube's or a random graph's is soon wide and better off with the
// grid: the search gives up (feature_block.cuh) and k_pdiam, launched behind it,
// does the work; that one leaves at once when this one has succeeded.
constexpr int kPdThreads = 1024;
constexpr int kPdSmem = 200 * 1024;
__global__ void __launch_bounds__(kPdThreads, 1) k_pdiam_block(BlockGraph g, BfsGraph q) {
  extern __shared__ __align__(16) unsigned char pd_smem[];
  if (block_status(q.ctl) != 0) return;
  g.c16 = q.ctl->col16;
  block_pdiam(g, q, pd_smem, kPdSmem);
}

__global__ void __launch_bounds__(kCgThreads, 1) k_pdiam(BfsGraph g, int32_t* d1, int32_t* d2,
                                                      int slot) {
  if (block_status(g.ctl) != 0 || g.ctl->pd_done) return;
  GridSync sync{g.ctl, slot, 0ull};
  const int tid = blockIdx.x * blockDim.x + threadIdx.x;
  pseudo_diameter_run(g, d1, d2, tid, gridDim.x * blockDim.x, sync);
}

__global__ void __launch_bounds__(kCgThreads, 1) k_bfs1(BfsGraph g, int32_t* dist, int src,
                                                     int slot) {
  if (block_status(g.ctl) != 0) return;
  GridSync sync{g.ctl, slot, 0ull};
  const int tid = blockIdx.x * blockDim.x + threadIdx.x;
  bfs_run(g, dist, kSrcSingle, src, kRoleFirst, tid, gridDim.x * blockDim.x, sync);
}

__global__ void k_copy_pdiam(const Ctl* c, int32_t* out) {
  const bool ok = c->status == 0;
  out[0] = ok ? c->pdiam : -1;
  out[1] = ok ? c->far_t : -1;
}

BfsGraph bfs_graph(const Launch& L) {
  BfsGraph g{};
  g.ctl = L.ws.ctl;
  g.rp = L.A->row_ptr;
  g.col = L.A->col;
  g.n = L.d.n;
  g.fq0 = L.ws.fq0;
  g.fq1 = L.ws.fq1;
  g.fq2 = L.ws.fq2;
  g.fq3 = L.ws.fq3;
  g.label = L.ws.label;
  g.ckey = L.ws.ckey;
  return g;
}

const void* bfs_kernel() { return (const void*)k_pdiam; }

cudaError_t launch_pseudo_diameter(const Launch& L, int slot, int starts) {
  BfsGraph g = bfs_graph(L);
  // (repeated searches, and a grid asked for, keep to the grid-wide kernel)
  if (L.d.n <= kPdMaxN && starts <= 1 && L.grid_req == 0) {
    cudaError_t e = cudaFuncSetAttribute(k_pdiam_block, cudaFuncAttributeMaxDynamicSharedMemorySize, kPdSmem);
    if (e != cudaSuccess) return e;
    const BlockGraph b{L.A->row_ptr, L.A->col, L.ws.slice_ptr, L.ws.slice_w, L.ws.scol, L.d.n, 0};
    k_pdiam_block<<<1, kPdThreads, kPdSmem, L.st>>>(b, g);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  int32_t* d1 = L.ws.dist;
  int32_t* d2 = L.ws.dist2;
  void* args[] = {&g, &d1, &d2, &slot};
  return cudaLaunchCooperativeKernel((const void*)k_pdiam, dim3(L.grid), dim3(kCgThreads), args, 0,
                                    L.st);
}

cudaError_t launch_bfs_only(const Launch& L, int src, int32_t* dist, int slot) {
  BfsGraph g = bfs_graph(L);
  void* args[] = {&g, &dist, &src, &slot};
  return cudaLaunchCooperativeKernel((const void*)k_bfs1, dim3(L.grid), dim3(kCgThreads), args, 0,
                                    L.st);
}

cudaError_t launch_copy_pdiam(const Launch& L, int32_t* out) {
  k_copy_pdiam<<<1, 1, 0, L.st>>>(L.ws.ctl, out);
  return cudaGetLastError();
}

}  // namespace mpcg
