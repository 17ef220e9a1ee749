// Dense layers of Eq. (NN) on CUDA cores (dense.cu): one launch covers every net of a layer.
#pragma once
#include "dp_internal.cuh"

namespace dpgb {

constexpr int kMaxDenseGroups = DP_MAX_TYPES * DP_MAX_TYPES;

// The rows that share one net: nrows consecutive rows from r0, or (with a row list) at most nrows
// entries of the list from r0, the number of which the device holds in DenseRows::count.
struct DenseGroup {
  long r0;
  long w;     // offset of W [n_in][n_out] in the parameter array; b follows W
  int nrows;
};
struct DenseRows {
  int ngroups = 0;
  const int* list = nullptr;   // row of every list entry, or null: consecutive rows
  const int* count = nullptr;  // device [ngroups], list mode only
  DenseGroup g[kMaxDenseGroups];
  void add(long r0, int nrows, long w) { g[ngroups++] = DenseGroup{r0, w, nrows}; }
  // rows of group k; a list holds at most nrows entries whatever was counted (append_row)
  __device__ __forceinline__ int rows_of(int k) const {
    return list ? min(__ldg(count + k), g[k].nrows) : g[k].nrows;
  }
};

// Row lists of a descriptor part: the slot rows with s != 0 (the others are padding) of every
// (centre type, neighbour type) pair, compacted so that no layer works on padding.  Entries of pair
// (ti, tj) start at base[ti * ntypes + tj], and there is room for cap[ti * ntypes + tj] of them.
// The room follows the per-type counts the call was set up with.  A device type array may have been rewritten
// since those were read: that is found on the device and the call is done again, but its kernels run to the
// end first, so entries beyond a pair's room are dropped.
struct RowLists {
  int* list = nullptr;
  int* count = nullptr;
  long base[kMaxDenseGroups];
  int cap[kMaxDenseGroups];
};

// Append every calling thread's row (grp in [0, ngroups)) to its group's list; the whole block calls.  One
// global atomic per block and group, so the order of a list differs from run to run: for layers whose rows
// do not meet in a sum.
__device__ __forceinline__ void append_row(const RowLists& rl, int ngroups, int grp, long row) {
  __shared__ int s_cnt[kMaxDenseGroups], s_base[kMaxDenseGroups];
  for (int e = threadIdx.x; e < ngroups; e += blockDim.x) s_cnt[e] = 0;
  if (grp >= ngroups) grp = -1;
  __syncthreads();
  const unsigned lane = threadIdx.x & 31u;
  const unsigned peers = __match_any_sync(0xffffffffu, grp);
  const int leader = __ffs(peers) - 1;
  int at = 0;
  if ((int)lane == leader && grp >= 0) at = atomicAdd(&s_cnt[grp], __popc(peers));
  at = __shfl_sync(0xffffffffu, at, leader) + __popc(peers & ((1u << lane) - 1u));
  __syncthreads();
  for (int e = threadIdx.x; e < ngroups; e += blockDim.x)
    if (s_cnt[e] > 0) s_base[e] = atomicAdd(rl.count + e, s_cnt[e]);
  __syncthreads();
  if (grp >= 0 && s_base[grp] + at < rl.cap[grp]) rl.list[rl.base[grp] + s_base[grp] + at] = (int)row;
}

// Row stride of the activations of an inner layer of width w: whole 16-byte (FP32) or 32-byte (FP64)
// quads, so that the next layer copies its operands as vectors.
__host__ __device__ inline int dense_ld(int w) { return (w + 3) & ~3; }

// One layer: input width and row stride, output width and row stride, skip (0 none, 1 +x, 2 +{x,x})
// and activation (1 tanh, 0 linear).
struct DenseShape {
  int n_in, ldx, n_out, ldy, skip, act;
};

// Y = phi(X W + b) + skip(X), T = phi(X W + b)
template <class R>
cudaError_t launch_dense_fwd(const DenseRows& rows, const DenseShape& s, const R* params, const R* X, R* Y, R* T,
                             cudaStream_t st);
// GX = (GY (1 - T^2)) W^T + skip^T(GY); s.act 0: no gate (T not read)
template <class R>
cudaError_t launch_dense_bwd(const DenseRows& rows, const DenseShape& s, const R* params, const R* GY, const R* T,
                             R* GX, cudaStream_t st);
// Forward and tangent: Y, T as above, Zd = Xd W, Yd = (1 - T^2) Zd + skip(Xd)  (tanh layers)
template <class R>
cudaError_t launch_dense_tan(const DenseRows& rows, const DenseShape& s, const R* params, const R* X, const R* Xd,
                             R* Y, R* T, R* Yd, R* Zd, cudaStream_t st);
// Reverse of that: GZd = GYd (1 - T^2), GZ = (GY - 2 T Zd GYd)(1 - T^2), GX = GZ W^T + skip^T(GY) and
// the same for the tangent pair; GZ and GZd are also written (the weight gradient reads them)
template <class R>
cudaError_t launch_dense_rev(const DenseRows& rows, const DenseShape& s, const R* params, const R* GY, const R* GYd,
                             const R* T, const R* Zd, R* GX, R* GXd, R* GZ, R* GZd, cudaStream_t st);

}  // namespace dpgb
