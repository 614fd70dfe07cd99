// knn.cu -- standalone kernel for the choice of eps1 by kNN (Sec. 11); the
// vote itself is knn_warp in knn_core.cuh.
#include "internal.h"
#include "knn_core.cuh"

namespace mpcg {

// q4: device query (n, m, l~, v); nullptr: take it from the control block.
// ctl nullable: then errors are reported as cls_out = -1, eps1_out = NaN.
__global__ void k_knn(KnnSpec s, Ctl* ctl, const double* q4, double* eps1_out,
                      int32_t* cls_out) {
  if (ctl && volatile_status(ctl) != 0) return;
  double chi[4];
  if (q4) {
    for (int c = 0; c < 4; ++c) chi[c] = q4[c];
  } else {
    chi[0] = (double)ctl->n;
    chi[1] = (double)ctl->nnz;
    chi[2] = (double)ctl->pdiam;
    chi[3] = ctl->v;
  }
  const int t = knn_warp(s, chi);
  if (threadIdx.x != 0) return;
  if (t < 0) {
    if (ctl) set_status(ctl, MPCG_ERR_INVALID_ARG);
    if (cls_out) *cls_out = -1;
    if (eps1_out) *eps1_out = NAN;
  } else {
    if (ctl) {
      ctl->cls = t;
      ctl->eps1 = pow10_neg(t);
    }
    if (cls_out) *cls_out = t;
    if (eps1_out) *eps1_out = pow10_neg(t);
  }
  if (ctl) ctl->t_features = globaltimer();
}

KnnSpec knn_spec(const mpcg_sample_t& S, const mpcg_options_t& o) {
  KnnSpec s{};
  s.feat = S.feat;
  s.cls = S.cls;
  s.count = S.count;
  s.k = o.knn_k;
  s.weighted = o.weighted;
  s.mask = o.feat_mask;
  for (int c = 0; c < 4; ++c) {
    s.fmin[c] = S.fmin[c];
    s.fmax[c] = S.fmax[c];
  }
  return s;
}

// Many queries (the classification of a test set, Sec. 12): one warp per
// query, kKnnWarps queries of a block at a time.  chi: [count][4]; cls:
// [count]; nbr: [count][k] or null (the indices of the k nearest in selection
// order, -1 past the sample's size).
//
// The block scales the sample once (the FP64 divisions) into shared memory, a
// tile of points at a time, also in single precision.  A query's pass looks
// at the single-precision distances; only a group of 32 points of which one
// may be nearer than the k-th found so far is computed in double, so the
// FP64 pipe, which bounded the pass, sees a few groups a query.  Scaled
// values up to M in magnitude are off by at most 2^-24 M each in single
// precision, so a difference by 4 2^-24 M, and the sum of four squares, its
// roundings included, by less than 140 x 2^-24 M^2 < 1e-5 M^2: a point whose
// single-precision distance is above the k-th distance by more than that is
// not among the k nearest.  Past M = 1e15, or where a value is not finite,
// every point is computed in double.
// 4,800 queries, 1,260 points, k = 5, with neighbours: 0.118 ms, against 7.37
// by a pass of all distances, divisions included, for every neighbour.
constexpr int kKnnWarps = 16;
constexpr int kKnnTile = 4096;  // points of a tile: 32 + 16 bytes each
__global__ void __launch_bounds__(kKnnWarps * 32) k_knn_batch(KnnSpec s, const double* chi4, int count,
                                                              int32_t* cls, int32_t* nbr, int tile) {
  extern __shared__ __align__(16) unsigned char knn_smem[];
  double* pd = reinterpret_cast<double*>(knn_smem);          // [4][tile]
  float* pf = reinterpret_cast<float*>(pd + 4 * (size_t)tile);  // [4][tile]
  __shared__ unsigned s_max;  // bits of the largest scaled magnitude of the tile (as a float)
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const unsigned full = 0xffffffffu;
  const int ntiles = (s.count + tile - 1) / tile;
  const int k = s.k < s.count ? s.k : s.count;
  for (int q0 = blockIdx.x * kKnnWarps; q0 < count; q0 += gridDim.x * kKnnWarps) {  // block-uniform
    const int qi = q0 + warp;
    double chi[4] = {0.0, 0.0, 0.0, 0.0}, q[4];
    if (qi < count)
      for (int c = 0; c < 4; ++c) chi[c] = chi4[4 * (size_t)qi + c];
    const bool good = knn_query(s, chi, q);
    float qf[4];
    unsigned qmax = __float_as_uint(1.0f);
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      qf[c] = (s.mask >> c) & 1u ? (float)q[c] : 0.0f;
      qmax = max(qmax, __float_as_uint(fabsf(qf[c])));  // NaN and infinity compare as largest
    }
    KnnList L;
    knn_clear(L);
    unsigned long long td = 0x7ff0000000000000ull;
    int ti = 0x7fffffff, bad = 0;
    for (int tl = 0; tl < ntiles; ++tl) {
      const int t0 = tl * tile, m = min(tile, s.count - t0);
      if (ntiles > 1 || q0 == blockIdx.x * kKnnWarps) {  // one tile stays for every query
        __syncthreads();
        if (threadIdx.x == 0) s_max = 0u;
        __syncthreads();
        unsigned mx = 0u;
        for (int e = threadIdx.x; e < 4 * m; e += blockDim.x) {
          const int c = e & 3, i = e >> 2;  // coalesced over the sample's rows
          // (a constant component, and one that is not selected, maps to 0)
          const double p = (s.mask >> c) & 1u
                               ? knn_scale(s.feat[4 * (size_t)t0 + e], s.fmin[c], s.fmax[c]) : 0.0;
          const float f = (float)p;
          pd[c * tile + i] = p;
          pf[c * tile + i] = f;
          mx = max(mx, __float_as_uint(fabsf(f)));
        }
        mx = __reduce_max_sync(full, mx);
        if (lane == 0) atomicMax(&s_max, mx);
        __syncthreads();
      }
      if (qi >= count || !good) continue;
      const unsigned mb = max(qmax, s_max);
      const float M = __uint_as_float(mb);
      const bool filter = mb < 0x7f800000u && M <= 1e15f;
      const float slack = 1e-5f * M * M;
      for (int base = 0; base < m; base += 32) {
        const int i = base + lane;
        const bool have = i < m;
        if (filter) {
          float df = 0.0f;
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            const float d = qf[c] - (have ? pf[c * tile + i] : 0.0f);
            df = __fmaf_rn(d, d, df);
          }
          const float lim = __double2float_ru(__longlong_as_double((long long)td)) + slack;
          if (!__any_sync(full, have && df <= lim)) continue;
        }
        double d2 = 0.0;
        if (have) {
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            if (!((s.mask >> c) & 1u)) continue;
            const double diff = __dsub_rn(q[c], pd[c * tile + i]);
            d2 = __dadd_rn(d2, __dmul_rn(diff, diff));
          }
        }
        if (d2 != d2) bad = 1;
        knn_enter(L, have, d2, t0 + i, k, td, ti);
      }
    }
    if (qi >= count) continue;
    const bool voted = good && !__any_sync(full, bad);
    const int t = voted ? knn_vote(s, L, k) : -1;
    if (lane == 0) cls[qi] = t;
    if (nbr) {
      int32_t* out = nbr + (size_t)qi * s.k;
      for (int j = lane; j < s.k; j += 32)
        out[j] = good && j < k ? (j < 32 ? L.i_lo : L.i_hi) : -1;
    }
  }
}

cudaError_t launch_knn_batch(cudaStream_t st, const mpcg_sample_t& S, const mpcg_options_t& o,
                             const double* chi4, int count, int32_t* cls, int32_t* nbr) {
  if (count <= 0) return cudaSuccess;
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return cudaErrorUnknown;
  // whole warps of points; a larger sample takes several tiles
  const int tile = S.count < kKnnTile ? (S.count + 31) / 32 * 32 : kKnnTile;
  const size_t smem = (size_t)tile * 4 * (sizeof(double) + sizeof(float));
  cudaError_t e = cudaFuncSetAttribute(k_knn_batch, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       kKnnTile * 4 * (int)(sizeof(double) + sizeof(float)));
  if (e != cudaSuccess) return e;
  const int need = (count + kKnnWarps - 1) / kKnnWarps;
  const int grid = need < sms ? need : sms;  // one scaled copy of the sample an SM
  k_knn_batch<<<grid, kKnnWarps * 32, smem, st>>>(knn_spec(S, o), chi4, count, cls, nbr, tile);
  return cudaGetLastError();
}

cudaError_t launch_knn(cudaStream_t st, const double* feat4, const mpcg_sample_t& S,
                       const mpcg_options_t& o, Ctl* ctl, double* eps1_out, int32_t* cls_out) {
  k_knn<<<1, 32, 0, st>>>(knn_spec(S, o), ctl, feat4, eps1_out, cls_out);
  return cudaGetLastError();
}

}  // namespace mpcg
