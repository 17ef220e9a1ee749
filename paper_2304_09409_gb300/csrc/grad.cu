// Parameter gradient of an energy + force objective (Sec. II.B, loss function):
//
//   Phi(theta) = sum_f a_f E_f + sum_i w_i . F_i = sum_f a_f E_f - D_w E,
//
// where D_w E is the derivative of E along the coordinate direction w.  For the loss
//   L = (1/B) sum_f [ pE dE_f^2 / N_f + pF sum_i |dF_i|^2 / (3 N_f) ]
// the caller passes a_f = 2 pE dE_f / (N_f B) and w_i = 2 pF dF_i / (3 N_f B), and dPhi/dtheta
// is dL/dtheta.  This is the "double backward" of the force: a tangent pass along w through
// every step (pair geometry, embedding, descriptor, fitting) gives D_w E; a reverse pass over
// both the primal and the tangent computation then gives the gradient with respect to every
// weight and bias.  Everything runs on CUDA cores in the model's precision (FP32 or FP64) with
// accumulation in the same precision; there is no framework autograd underneath.
//
// Dense layer (Eq. (NN)) with tangent:  z = x W + b, t = tanh z, y = t + skip(x)
//                                       zd = xd W,  yd = (1 - t^2) zd + skip(xd)
// reverse, given gy = dPhi/dy and gyd = dPhi/dyd:
//   gzd = gyd (1 - t^2);  gz = (gy - 2 t zd gyd) (1 - t^2)
//   gx = gz W^T + skip^T(gy);  gxd = gzd W^T + skip^T(gyd);  gW += x^T gz + xd^T gzd;  gb += sum gz
#include <cstring>

#include "capi_internal.cuh"
#include "dense.cuh"
#include "env.cuh"
#include "grad.cuh"

namespace dpgb {

namespace {

inline unsigned nb(long n, int b) { return (unsigned)((n + b - 1) / b); }
inline int net_index(const PathConst& pc, int ti, int tj) { return pc.type_one_side ? tj : ti * pc.ntypes + tj; }

// ---- row lists in row order -------------------------------------------------------------------
// The weight gradient sums along the lists, so here their order is fixed: every block of kListThreads rows counts
// its rows of every type pair, the counts are scanned, and each row is written at its place.  (The forward passes
// take their lists from append_row: no result depends on that order.)  Three small launches for one;
// 6,144 atoms of 138 slots: 8.54 ms a training step against 8.52.
constexpr int kListThreads = 256;

// Rows of group grp among the threads of lower number (grp < 0: none), and in s_base[group] those of the whole
// block.  The whole block calls.
__device__ __forceinline__ int rank_in_block(int ngroups, int grp, int* s_base) {
  __shared__ int s_warp[kListThreads / 32][kMaxDenseGroups];
  const unsigned lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
  for (int e = threadIdx.x; e < (kListThreads / 32) * kMaxDenseGroups; e += kListThreads) (&s_warp[0][0])[e] = 0;
  __syncthreads();
  const unsigned peers = __match_any_sync(0xffffffffu, grp);
  if (grp >= 0 && (int)lane == __ffs(peers) - 1) s_warp[warp][grp] = __popc(peers);
  __syncthreads();
  for (int g = threadIdx.x; g < ngroups; g += kListThreads) {
    int at = 0;
    for (int w = 0; w < kListThreads / 32; ++w) {
      const int n = s_warp[w][g];
      s_warp[w][g] = at;
      at += n;
    }
    s_base[g] = at;
  }
  __syncthreads();
  return grp >= 0 ? s_warp[warp][grp] + __popc(peers & ((1u << lane) - 1u)) : 0;
}
// block_count [ngroups][blocks]
__device__ __forceinline__ void count_rows(int ngroups, int grp, int* __restrict__ block_count) {
  __shared__ int s_total[kMaxDenseGroups];
  rank_in_block(ngroups, grp, s_total);
  for (int g = threadIdx.x; g < ngroups; g += kListThreads)
    block_count[(long)g * gridDim.x + blockIdx.x] = s_total[g];
}
// Exclusive scan of a group's block counts, in place, and its total; a block per group.
__global__ void __launch_bounds__(1024) k_scan_rows(int* __restrict__ block_count, int nblocks, int* __restrict__ count) {
  __shared__ int s_sum[32];
  int* c = block_count + (long)blockIdx.x * nblocks;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int per = (nblocks + 1023) / 1024, b0 = min(nblocks, (int)threadIdx.x * per), b1 = min(nblocks, b0 + per);
  int sum = 0;
  for (int b = b0; b < b1; ++b) sum += c[b];
  int incl = sum;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const int x = __shfl_up_sync(0xffffffffu, incl, off);
    if (lane >= off) incl += x;
  }
  if (lane == 31) s_sum[warp] = incl;
  __syncthreads();
  int at = incl - sum;
  for (int w = 0; w < warp; ++w) at += s_sum[w];
  for (int b = b0; b < b1; ++b) {
    const int n = c[b];
    c[b] = at;
    at += n;
  }
  if (threadIdx.x == 1023) count[blockIdx.x] = at;
}
// The rows at their places (those beyond a pair's room are dropped, as append_row drops them).
template <class R>
__global__ void __launch_bounds__(kListThreads)
    k_fill_rows(PathConst pc, const R* __restrict__ Renv, const int* __restrict__ tsorted,
                const int* __restrict__ block_start, RowLists rl) {
  __shared__ int s_total[kMaxDenseGroups];
  const long row = (long)blockIdx.x * kListThreads + threadIdx.x;
  int grp = -1;
  if (row < (long)pc.natoms * pc.nc && Renv[row * 4] != R(0))
    grp = tsorted[row / pc.nc] * pc.ntypes + slot_block(pc, (int)(row % pc.nc));
  const int rank = rank_in_block(pc.ntypes * pc.ntypes, grp, s_total);
  if (grp < 0) return;
  const int at = block_start[(long)grp * gridDim.x + blockIdx.x] + rank;
  if (at < rl.cap[grp]) rl.list[rl.base[grp] + at] = (int)row;
}

// ---- pair geometry and its tangent along w -----------------------------------------------------
template <class R>
__global__ void k_env_tan(PathConst pc, const double* __restrict__ coord, const double* __restrict__ w,
                          const double* __restrict__ gv, const int* __restrict__ perm, const int* __restrict__ nl_j,
                          const int* __restrict__ nl_code, const int* __restrict__ tsorted,
                          int* __restrict__ block_count, R* __restrict__ Renv, R* __restrict__ Rdot) {
  const long row = (long)blockIdx.x * blockDim.x + threadIdx.x;
  const bool in = row < (long)pc.natoms * pc.nc;
  const int p = in ? (int)(row / pc.nc) : 0, k = in ? (int)(row % pc.nc) : 0;
  const int i = perm[p];
  const int j = in ? nl_j[(long)i * pc.nc + k] : -1;
  R o[4] = {0, 0, 0, 0}, od[4] = {0, 0, 0, 0};
  if (j >= 0) {
    double d0, d1, d2;
    listed_disp(coord + 3 * i, coord + 3 * j, nl_code[(long)i * pc.nc + k], pc, frame_of(pc, i), d0, d1, d2);
    R r, s, ds, u[3];
    pair_env<R>(d0, d1, d2, norm2_exact(d0, d1, d2), pc.rs, pc.rc, pc.near2, r, s, ds, u);
    // dd = (w_j - w_i) + g_f r_ij (the virial seed of the frame: sum_ab g_ab Xi_ab is minus the
    // derivative of E along the homogeneous deformation r_ij -> r_ij + g r_ij); dr = u . dd;
    // du = (dd - dr u) / r; ds/de = s' dr
    double e0 = w[3 * j] - w[3 * i], e1 = w[3 * j + 1] - w[3 * i + 1], e2 = w[3 * j + 2] - w[3 * i + 2];
    if (gv) {
      const double* g = gv + 9L * frame_of(pc, i);
      e0 += g[0] * d0 + g[1] * d1 + g[2] * d2;
      e1 += g[3] * d0 + g[4] * d1 + g[5] * d2;
      e2 += g[6] * d0 + g[7] * d1 + g[8] * d2;
    }
    const R dd[3] = {R(e0), R(e1), R(e2)};
    const R dr = u[0] * dd[0] + u[1] * dd[1] + u[2] * dd[2];
    const R sd = ds * dr;
    o[0] = s;
    od[0] = sd;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const R ud = (dd[a] - dr * u[a]) / r;
      o[1 + a] = s * u[a];
      od[1 + a] = sd * u[a] + s * ud;
    }
  }
  if (in)
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      Renv[row * 4 + a] = o[a];
      Rdot[row * 4 + a] = od[a];
    }
  // rows the embedding layers work on: this block's number of them, by type pair
  count_rows(pc.ntypes * pc.ntypes, o[0] != R(0) ? tsorted[p] * pc.ntypes + slot_block(pc, k) : -1, block_count);
}

// ---- first embedding layer (scalar input), primal and tangent ----------------------------------
template <class R>
__global__ void k_emb0_tan(PathConst pc, NetPtrs<R> nets, const int* __restrict__ tsorted, const R* __restrict__ Renv,
                           const R* __restrict__ Rdot, int w1, int ld, int skip, R* __restrict__ Y, R* __restrict__ T,
                           R* __restrict__ Yd, R* __restrict__ Zd) {
  const long e = (long)blockIdx.x * blockDim.x + threadIdx.x;
  const long nrow = (long)pc.natoms * pc.nc;
  if (e >= nrow * w1) return;
  const long row = e / w1;
  const int o = (int)(e % w1);
  const int p = (int)(row / pc.nc), k = (int)(row % pc.nc);
  const int net = net_of(pc, tsorted[p], slot_block(pc, k));
  const R s = Renv[row * 4], sd = Rdot[row * 4];
  if (s == R(0)) return;  // padding: in no row list, read by nobody
  const R wv = nets.w0[net][o];
  const R t = tanh_r(s * wv + nets.b0[net][o]);
  const R zd = sd * wv;
  const long at = row * ld + o;
  Y[at] = t + (skip ? s : R(0));
  T[at] = t;
  Zd[at] = zd;
  Yd[at] = (R(1) - t * t) * zd + (skip ? sd : R(0));
}

// ---- weight and bias gradients: gW += X^T GZ + Xd^T GZd, gb += sum_rows GZ ----------------------
// One launch covers every net of a layer.  One block owns a 64 x 64 tile of one net's gW and a slab of
// its rows (a range, or entries of the row list) and sums them in order; the slabs' sums go to gW with atomics.  128 threads keep
// 8 x 4 outputs each (FP32: six 16-byte shared loads per 64 FMAs); the next 16 rows' global loads are
// in flight while the current ones are summed.  Bound by FP32 FMAs and those loads: the 6,144-atom batch's
// layers 3.65 -> 1.63 ms.
template <class R>
struct WGradJob {
  DenseRows rows;
  int slab0[kMaxDenseGroups];  // first slab of every net
  int slab_rows[kMaxDenseGroups];
  int n_in, ldx, n_out, ldg;
  const R *X, *Xd, *GZ, *GZd;
  R* grad;  // gW at the net's parameter offset, gb behind it
};

constexpr int kWgTI = 64, kWgRR = 16, kWgThreads = 128, kWgLd = kWgTI + 4;

template <class R>
__global__ void __launch_bounds__(kWgThreads)
    k_wgrad(const __grid_constant__ WGradJob<R> g) {
  constexpr int TI = kWgTI, RR = kWgRR, NT = kWgThreads, LD = kWgLd;
  constexpr int PER = RR * TI / NT;  // values per thread, array and step
  __shared__ __align__(32) R xs[2][RR][LD], gs[2][RR][LD];  // primal and tangent rows
  using Q = typename Vec4<R>::T;
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;  // outputs i = 8 ty + a, o = 4 tx + b
  const int i0 = blockIdx.x * TI, o0 = blockIdx.y * TI;
  int gi = 0;
  while (gi + 1 < g.rows.ngroups && (int)blockIdx.z >= g.slab0[gi + 1]) ++gi;
  const DenseGroup grp = g.rows.g[gi];
  const int nrows = g.rows.rows_of(gi);
  const int rbeg = ((int)blockIdx.z - g.slab0[gi]) * g.slab_rows[gi];
  const int rend = min(nrows, rbeg + g.slab_rows[gi]);
  if (rbeg >= rend) return;
  R acc[8][4] = {}, bacc[4] = {};
  // thread tid loads column tid % 64 of rows tid / 64 + 2 q
  const int lc = tid % TI, lr = tid / TI;
  R px[PER], pxd[PER], pg[PER], pgd[PER];
  auto row_of = [&](int r) -> long {
    if (r >= rend) return -1;
    return g.rows.list ? __ldg(g.rows.list + grp.r0 + r) : grp.r0 + r;
  };
  long nrow[PER];
  auto rows_of = [&](int r0) {
#pragma unroll
    for (int q = 0; q < PER; ++q) nrow[q] = row_of(r0 + lr + 2 * q);
  };
  auto fetch = [&]() {
#pragma unroll
    for (int q = 0; q < PER; ++q) {
      const long row = nrow[q];
      const bool xv = row >= 0 && i0 + lc < g.n_in, gv = row >= 0 && o0 + lc < g.n_out;
      px[q] = xv ? g.X[row * g.ldx + i0 + lc] : R(0);
      pxd[q] = xv ? g.Xd[row * g.ldx + i0 + lc] : R(0);
      pg[q] = gv ? g.GZ[row * g.ldg + o0 + lc] : R(0);
      pgd[q] = gv ? g.GZd[row * g.ldg + o0 + lc] : R(0);
    }
  };
  rows_of(rbeg);
  fetch();
  rows_of(rbeg + RR);
  for (int r0 = rbeg; r0 < rend; r0 += RR) {
    __syncthreads();  // the previous rows were read
#pragma unroll
    for (int q = 0; q < PER; ++q) {
      const int r = lr + 2 * q;
      xs[0][r][lc] = px[q];
      xs[1][r][lc] = pxd[q];
      gs[0][r][lc] = pg[q];
      gs[1][r][lc] = pgd[q];
    }
    __syncthreads();
    if (r0 + RR < rend) {
      fetch();
      rows_of(r0 + 2 * RR);
    }
#pragma unroll 4
    for (int r = 0; r < RR; ++r) {
      const Q g4 = *reinterpret_cast<const Q*>(&gs[0][r][tx * 4]), gd4 = *reinterpret_cast<const Q*>(&gs[1][r][tx * 4]);
      const R ga[4] = {g4.x, g4.y, g4.z, g4.w}, gda[4] = {gd4.x, gd4.y, gd4.z, gd4.w};
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const Q x4 = *reinterpret_cast<const Q*>(&xs[0][r][ty * 8 + 4 * h]);
        const Q xd4 = *reinterpret_cast<const Q*>(&xs[1][r][ty * 8 + 4 * h]);
        const R xa[4] = {x4.x, x4.y, x4.z, x4.w}, xda[4] = {xd4.x, xd4.y, xd4.z, xd4.w};
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
          for (int b = 0; b < 4; ++b) acc[4 * h + a][b] += xa[a] * ga[b] + xda[a] * gda[b];
      }
      if (blockIdx.x == 0 && ty == 0)
#pragma unroll
        for (int b = 0; b < 4; ++b) bacc[b] += ga[b];
    }
  }
  R* gW = g.grad + grp.w;
#pragma unroll
  for (int a = 0; a < 8; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      const int i = i0 + ty * 8 + a, o = o0 + tx * 4 + b;
      if (i < g.n_in && o < g.n_out) atomicAdd(gW + (long)i * g.n_out + o, acc[a][b]);
    }
  if (blockIdx.x == 0 && ty == 0)
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      const int o = o0 + tx * 4 + b;
      if (o < g.n_out) atomicAdd(gW + (long)g.n_in * g.n_out + o, bacc[b]);
    }
}

// ---- first embedding layer reverse and its weight/bias gradients (all nets) ----------------------
template <class R>
__global__ void __launch_bounds__(256)
    k_emb0_rev(PathConst pc, const int* __restrict__ tsorted, const R* __restrict__ Renv, const R* __restrict__ Rdot,
               int w1, int ld, const R* __restrict__ GY, const R* __restrict__ GYd, const R* __restrict__ T,
               const R* __restrict__ Zd, long rows_per_block, R* __restrict__ grad, NetOffsets off) {
  extern __shared__ __align__(16) unsigned char sm_raw[];
  R* acc = reinterpret_cast<R*>(sm_raw);  // [nets][w1][2] (gw, gb)
  const int nets = off.nets;
  for (int e = threadIdx.x; e < nets * w1 * 2; e += blockDim.x) acc[e] = R(0);
  __syncthreads();
  const long nrow = (long)pc.natoms * pc.nc;
  const long beg = blockIdx.x * rows_per_block, end = min(nrow, beg + rows_per_block);
  for (long e = beg * w1 + threadIdx.x; e < end * w1; e += blockDim.x) {
    const long row = e / w1;
    const int o = (int)(e % w1);
    const int p = (int)(row / pc.nc), k = (int)(row % pc.nc);
    const int net = net_of(pc, tsorted[p], slot_block(pc, k));
    const R s = Renv[row * 4], sd = Rdot[row * 4];
    if (s == R(0)) continue;  // padding
    const long at = row * ld + o;
    const R t = T[at], g = R(1) - t * t;
    const R gyd = GYd[at];
    const R gzd = gyd * g;
    const R gz = (GY[at] - R(2) * t * Zd[at] * gyd) * g;
    atomicAdd(acc + (net * w1 + o) * 2, s * gz + sd * gzd);
    atomicAdd(acc + (net * w1 + o) * 2 + 1, gz);
  }
  __syncthreads();
  for (int e = threadIdx.x; e < nets * w1; e += blockDim.x) {
    const int net = e / w1, o = e % w1;
    atomicAdd(grad + off.w[net] + o, acc[e * 2]);
    atomicAdd(grad + off.w[net] + w1 + o, acc[e * 2 + 1]);
  }
}

// ---- T, Td, D, Dd per atom --------------------------------------------------------------------
template <class R>
__global__ void k_contract_tan(PathConst pc, const R* __restrict__ G, const R* __restrict__ Gd,
                               const R* __restrict__ Renv, const R* __restrict__ Rdot, R* __restrict__ Tm,
                               R* __restrict__ Tmd, R* __restrict__ D, R* __restrict__ Dd) {
  extern __shared__ __align__(16) unsigned char sm_raw[];
  const int M = pc.M, A = pc.A, nc = pc.nc;
  R* Ts = reinterpret_cast<R*>(sm_raw);
  R* Tds = Ts + M * 4;
  const int p = blockIdx.x;
  const R inv = R(1) / R(nc);
  for (int m = threadIdx.x; m < M; m += blockDim.x) {
    R a[4] = {0, 0, 0, 0}, ad[4] = {0, 0, 0, 0};
    for (int t = 0; t < pc.ntypes; ++t)
      for (int k = pc.sel_off[t]; k < pc.sel_off[t + 1]; ++k) {
        const long row = (long)p * nc + k;
        const typename Vec4<R>::T rr = reinterpret_cast<const typename Vec4<R>::T*>(Renv)[row];
        if (rr.x == R(0)) break;  // the zero rows close each type block; nothing is computed for them
        const typename Vec4<R>::T rd = reinterpret_cast<const typename Vec4<R>::T*>(Rdot)[row];
        const R g = G[row * M + m], gd = Gd[row * M + m];
        a[0] += g * rr.x;
        a[1] += g * rr.y;
        a[2] += g * rr.z;
        a[3] += g * rr.w;
        ad[0] += gd * rr.x + g * rd.x;
        ad[1] += gd * rr.y + g * rd.y;
        ad[2] += gd * rr.z + g * rd.z;
        ad[3] += gd * rr.w + g * rd.w;
      }
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      Ts[m * 4 + c] = a[c] * inv;
      Tds[m * 4 + c] = ad[c] * inv;
      Tm[((long)p * M + m) * 4 + c] = a[c] * inv;
      Tmd[((long)p * M + m) * 4 + c] = ad[c] * inv;
    }
  }
  __syncthreads();
  for (int idx = threadIdx.x; idx < M * A; idx += blockDim.x) {
    const int m = idx / A, l = idx % A;
    R v = 0, vd = 0;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      v += Ts[m * 4 + c] * Ts[l * 4 + c];
      vd += Tds[m * 4 + c] * Ts[l * 4 + c] + Ts[m * 4 + c] * Tds[l * 4 + c];
    }
    D[(long)p * M * A + idx] = v;
    Dd[(long)p * M * A + idx] = vd;
  }
}

// ---- dPhi/dT, dPhi/dTd from dPhi/dD, dPhi/dDd; then dPhi/dG, dPhi/dGd per slot -------------------
template <class R>
__global__ void k_descr_rev(PathConst pc, const R* __restrict__ Tm, const R* __restrict__ Tmd,
                            const R* __restrict__ gD, const R* __restrict__ gDd, const R* __restrict__ Renv,
                            const R* __restrict__ Rdot, R* __restrict__ gG, R* __restrict__ gGd) {
  extern __shared__ __align__(16) unsigned char sm_raw[];
  const int M = pc.M, A = pc.A, nc = pc.nc;
  R* Ts = reinterpret_cast<R*>(sm_raw);
  R* Tds = Ts + M * 4;
  R* gTs = Tds + M * 4;
  R* gTds = gTs + M * 4;
  const int p = blockIdx.x;
  for (int e = threadIdx.x; e < M * 4; e += blockDim.x) {
    Ts[e] = Tm[(long)p * M * 4 + e];
    Tds[e] = Tmd[(long)p * M * 4 + e];
  }
  __syncthreads();
  const R* gDp = gD + (long)p * M * A;
  const R* gDdp = gDd + (long)p * M * A;
  for (int e = threadIdx.x; e < M * 4; e += blockDim.x) {
    const int m = e >> 2, c = e & 3;
    R gt = 0, gtd = 0;
    for (int l = 0; l < A; ++l) {
      gt += gDp[m * A + l] * Ts[l * 4 + c] + gDdp[m * A + l] * Tds[l * 4 + c];
      gtd += gDdp[m * A + l] * Ts[l * 4 + c];
    }
    if (m < A)
      for (int q = 0; q < M; ++q) {
        gt += gDp[q * A + m] * Ts[q * 4 + c] + gDdp[q * A + m] * Tds[q * 4 + c];
        gtd += gDdp[q * A + m] * Ts[q * 4 + c];
      }
    gTs[e] = gt;
    gTds[e] = gtd;
  }
  __syncthreads();
  const R inv = R(1) / R(nc);
  for (int e = threadIdx.x; e < nc * M; e += blockDim.x) {
    const int k = e / M, m = e % M;
    const long row = (long)p * nc + k;
    if (Renv[row * 4] == R(0)) continue;  // padding: in no row list
    R g = 0, gd = 0;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const R rr = Renv[row * 4 + c], rd = Rdot[row * 4 + c];
      g += gTs[m * 4 + c] * rr + gTds[m * 4 + c] * rd;
      gd += gTds[m * 4 + c] * rr;
    }
    gG[row * M + m] = g * inv;
    gGd[row * M + m] = gd * inv;
  }
}

// ---- last (linear) fitting layer reverse: seeds a_f (energy) and -1 (tangent) ------------------
template <class R>
__global__ void k_fit_last_rev(int n, const int* __restrict__ perm, const int* __restrict__ atom_frame,
                               const double* __restrict__ a_frame, double b, const R* __restrict__ wl, int n_in,
                               R* __restrict__ gx, R* __restrict__ gxd, R* __restrict__ gz, R* __restrict__ gzd) {
  const long e = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= (long)n * n_in) return;
  const int p = (int)(e / n_in), c = (int)(e % n_in);
  const int i = perm[p];
  const R a = (R)a_frame[atom_frame ? atom_frame[i] : 0];
  gx[e] = a * wl[c];
  gxd[e] = (R)b * wl[c];
  if (c == 0) {
    gz[p] = a;
    gzd[p] = (R)b;
  }
}

template <class R>
__global__ void k_to_double(const R* __restrict__ x, long n, double* __restrict__ y) {
  const long e = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (e < n) y[e] = (double)x[e];
}

__global__ void k_types_sorted(const int* __restrict__ type, const int* __restrict__ perm, int n, int ntypes,
                               int* __restrict__ out) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p < n) out[p] = type_in_range(type[perm[p]], ntypes);
}

template <class R>
__global__ void k_zero(R* __restrict__ x, long n) {
  const long e = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (e < n) x[e] = R(0);
}

template <class R>
void launch_wgrad(const DenseRows& rows, const DenseShape& sh, const R* X, const R* Xd, const R* GZ, const R* GZd,
                  int ldg, R* grad, cudaStream_t st) {
  WGradJob<R> g;
  std::memset(&g, 0, sizeof(g));
  g.rows = rows;
  g.n_in = sh.n_in;
  g.ldx = sh.ldx;
  g.n_out = sh.n_out;
  g.ldg = ldg;
  g.X = X;
  g.Xd = Xd;
  g.GZ = GZ;
  g.GZd = GZd;
  g.grad = grad;
  const long tiles = (long)nb(sh.n_in, kWgTI) * nb(sh.n_out, kWgTI);
  // Slabs of 4096 rows.  Consecutive rows (the fitting net) take shorter ones, down to 512, while a net's
  // launch leaves SMs under two blocks each: every slab is one FP32 chain per output, so long slabs keep
  // the number of atomics low.  Listed rows (the embedding nets, whose outputs are few tiles) go down to
  // 128 rows while the whole layer leaves SMs under eight blocks each.
  long most = 0;
  for (int k = 0; k < rows.ngroups; ++k) most += rows.g[k].nrows;
  int listed = 4096;
  while (listed > 128 && tiles * ((most + listed - 1) / listed) < 8L * sm_count()) listed /= 2;
  int at = 0;
  for (int k = 0; k < rows.ngroups; ++k) {
    int n = rows.list ? listed : 4096;
    if (!rows.list)
      while (n > 512 && tiles * nb(rows.g[k].nrows, n) < 2L * sm_count()) n /= 2;
    g.slab_rows[k] = n;
    g.slab0[k] = at;
    at += (rows.g[k].nrows + n - 1) / n;
  }
  if (at == 0) return;
  k_wgrad<R><<<dim3(nb(sh.n_in, kWgTI), nb(sh.n_out, kWgTI), at), kWgThreads, 0, st>>>(g);
}

}  // namespace

template <class R>
int run_grad(const DeviceModel& m, const PathConst& pc, const R* params, const PathIO& io, const double* w_dev,
             const double* a_dev, const double* gv_dev, double b, Arena& ar, cudaStream_t st, R** grad_out) {
  const long N = pc.natoms, nc = pc.nc, rows = N * nc;
  const int M = pc.M, A = pc.A, ne = m.cfg.n_embed, nfl = m.n_fit_layers, nt = pc.ntypes;
  // ---- scratch ----
  R* Renv = ar.get<R>(rows * 4);
  R* Rdot = ar.get<R>(rows * 4);
  // row stride of layer l's activations: the last layer's rows are read by the descriptor kernels
  auto emb_ld = [&](int l) { return l == ne - 1 ? m.cfg.embed[l] : dense_ld(m.cfg.embed[l]); };
  auto emb_shape = [&](int l) {
    const LayerDesc& L = m.emb[l];
    return DenseShape{L.n_in, emb_ld(l - 1), L.n_out, emb_ld(l), L.skip, 1};
  };
  auto fit_shape = [&](int l) {
    const LayerDesc& L = m.fit[l];
    return DenseShape{L.n_in, L.n_in, L.n_out, L.n_out, L.skip, L.tanh_act};
  };
  std::vector<R*> Ye(ne), Te(ne), Yed(ne), Zed(ne);
  int maxe = 1;
  for (int l = 0; l < ne; ++l) {
    const long wl = emb_ld(l);
    maxe = std::max(maxe, (int)wl);
    Ye[l] = ar.get<R>(rows * wl);
    Te[l] = ar.get<R>(rows * wl);
    Yed[l] = ar.get<R>(rows * wl);
    Zed[l] = ar.get<R>(rows * wl);
  }
  R* Tm = ar.get<R>(N * M * 4);
  R* Tmd = ar.get<R>(N * M * 4);
  R* D = ar.get<R>(N * M * A);
  R* Dd = ar.get<R>(N * M * A);
  std::vector<R*> Yf(nfl), Tf(nfl), Yfd(nfl), Zfd(nfl);
  int maxf = M * A;
  for (int l = 0; l < nfl; ++l) {
    const long wl = m.fit[l].n_out;
    maxf = std::max(maxf, (int)wl);
    Yf[l] = ar.get<R>(N * wl);
    Tf[l] = ar.get<R>(N * wl);
    Yfd[l] = ar.get<R>(N * wl);
    Zfd[l] = ar.get<R>(N * wl);
  }
  R* fa = ar.get<R>(N * maxf);
  R* fad = ar.get<R>(N * maxf);
  R* fb = ar.get<R>(N * maxf);
  R* fbd = ar.get<R>(N * maxf);
  R* fz = ar.get<R>(N * maxf);
  R* fzd = ar.get<R>(N * maxf);
  R* ea = ar.get<R>(rows * maxe);
  R* ead = ar.get<R>(rows * maxe);
  R* eb = ar.get<R>(rows * maxe);
  R* ebd = ar.get<R>(rows * maxe);
  R* ez = ar.get<R>(rows * maxe);
  R* ezd = ar.get<R>(rows * maxe);
  int* tsorted = ar.get<int>(N);
  R* grad = ar.get<R>(m.n_params);
  RowLists lists;
  lists.list = ar.get<int>(rows);
  lists.count = ar.get<int>(kMaxDenseGroups);
  const unsigned list_blocks = nb(rows, kListThreads);
  int* block_count = ar.get<int>((long)nt * nt * list_blocks);
  long list_at = 0;
  for (int ti = 0; ti < nt; ++ti)
    for (int tj = 0; tj < nt; ++tj) {
      lists.base[ti * nt + tj] = list_at;
      lists.cap[ti * nt + tj] = (io.type_start[ti + 1] - io.type_start[ti]) * pc.sel[tj];
      list_at += lists.cap[ti * nt + tj];
    }
  if (ar.measure) return DP_OK;
  if (!ar.ok()) {
    set_error("scratch allocation failed");
    return DP_E_OOM;
  }
  k_zero<R><<<nb(m.n_params, 256), 256, 0, st>>>(grad, m.n_params);
  k_types_sorted<<<nb(N, 256), 256, 0, st>>>(io.type, io.perm, (int)N, nt, tsorted);
  // ---- forward: primal and tangent ----
  {
    ProfScope _ps(io.prof, "grad_env", st, 3);
    k_env_tan<R><<<list_blocks, kListThreads, 0, st>>>(pc, io.coord, w_dev, gv_dev, io.perm, io.nl_j, io.nl_code,
                                                      tsorted, block_count, Renv, Rdot);
    k_scan_rows<<<nt * nt, 1024, 0, st>>>(block_count, (int)list_blocks, lists.count);
    k_fill_rows<R><<<list_blocks, kListThreads, 0, st>>>(pc, Renv, tsorted, block_count, lists);
  }
  NetPtrs<R> nets;
  NetOffsets off;
  off.nets = m.n_embed_nets;
  for (int n = 0; n < m.n_embed_nets; ++n) {
    const LayerDesc& L0 = m.emb[(size_t)n * ne];
    nets.w0[n] = params + L0.w_off;
    nets.b0[n] = params + L0.w_off + (long)L0.n_in * L0.n_out;
    off.w[n] = L0.w_off;
  }
  const int w1 = m.cfg.embed[0];
  k_emb0_tan<R><<<nb(rows * w1, 256), 256, 0, st>>>(pc, nets, tsorted, Renv, Rdot, w1, emb_ld(0), m.emb[0].skip, Ye[0], Te[0],
                                                     Yed[0], Zed[0]);
  auto emb_layer = [&](int l) {
    DenseRows r;
    r.list = lists.list;
    r.count = lists.count;
    for (int ti = 0; ti < nt; ++ti)
      for (int tj = 0; tj < nt; ++tj)
        r.add(lists.base[ti * nt + tj], (io.type_start[ti + 1] - io.type_start[ti]) * pc.sel[tj],
              m.emb[(size_t)net_index(pc, ti, tj) * ne + l].w_off);
    return r;
  };
  auto fit_layer = [&](int l) {
    DenseRows r;
    for (int t = 0; t < nt; ++t)
      r.add(io.type_start[t], io.type_start[t + 1] - io.type_start[t], m.fit[(size_t)t * nfl + l].w_off);
    return r;
  };
  for (int l = 1; l < ne; ++l) {
    ProfScope _ps(io.prof, "grad_emb_fwd", st);
    DP_CUDA_TRY(launch_dense_tan<R>(emb_layer(l), emb_shape(l), params, Ye[l - 1], Yed[l - 1], Ye[l], Te[l], Yed[l],
                                    Zed[l], st));
  }
  k_contract_tan<R><<<(unsigned)N, 128, sizeof(R) * M * 8, st>>>(pc, Ye[ne - 1], Yed[ne - 1], Renv, Rdot, Tm, Tmd, D,
                                                                   Dd);
  for (int l = 0; l < nfl - 1; ++l) {
    ProfScope _ps(io.prof, "grad_fit_fwd", st);
    DP_CUDA_TRY(launch_dense_tan<R>(fit_layer(l), fit_shape(l), params, l > 0 ? Yf[l - 1] : D, l > 0 ? Yfd[l - 1] : Dd,
                                    Yf[l], Tf[l], Yfd[l], Zfd[l], st));
  }
  // ---- reverse: fitting net ----
  {
    // per type (the output weights differ): gx = a w, gxd = b w at the last hidden output
    for (int t = 0; t < nt; ++t) {
      const int nrows = io.type_start[t + 1] - io.type_start[t];
      if (nrows <= 0) continue;
      const LayerDesc& L = m.fit[(size_t)t * nfl + nfl - 1];
      const long r0 = io.type_start[t];
      k_fit_last_rev<R><<<nb((long)nrows * L.n_in, 256), 256, 0, st>>>(
          nrows, io.perm + r0, pc.atom_frame, a_dev, b, params + L.w_off, L.n_in, fa + r0 * L.n_in, fad + r0 * L.n_in,
          fz + r0, fzd + r0);
    }
    // output layer weight/bias gradients: x = last hidden output, gz = a, gzd = b
    launch_wgrad<R>(fit_layer(nfl - 1), fit_shape(nfl - 1), nfl >= 2 ? Yf[nfl - 2] : D, nfl >= 2 ? Yfd[nfl - 2] : Dd,
                    fz, fzd, 1, grad, st);
  }
  R* gy = fa;
  R* gyd = fad;
  R* gx = fb;
  R* gxd = fbd;
  for (int l = nfl - 2; l >= 0; --l) {
    {
      ProfScope _ps(io.prof, "grad_fit_rev", st);
      DP_CUDA_TRY(launch_dense_rev<R>(fit_layer(l), fit_shape(l), params, gy, gyd, Tf[l], Zfd[l], gx, gxd, fz, fzd, st));
    }
    ProfScope _ps(io.prof, "grad_fit_w", st);
    launch_wgrad<R>(fit_layer(l), fit_shape(l), l > 0 ? Yf[l - 1] : D, l > 0 ? Yfd[l - 1] : Dd, fz, fzd, m.fit[l].n_out,
                    grad, st);
    std::swap(gy, gx);
    std::swap(gyd, gxd);
  }
  // gy, gyd now hold dPhi/dD, dPhi/dDd
  {
    const size_t sm = sizeof(R) * M * 16;
    k_descr_rev<R><<<(unsigned)N, 128, sm, st>>>(pc, Tm, Tmd, gy, gyd, Renv, Rdot, ea, ead);
  }
  // ---- reverse: embedding nets ----
  R* egy = ea;
  R* egyd = ead;
  R* egx = eb;
  R* egxd = ebd;
  for (int l = ne - 1; l >= 1; --l) {
    {
      ProfScope _ps(io.prof, "grad_emb_rev", st);
      DP_CUDA_TRY(launch_dense_rev<R>(emb_layer(l), emb_shape(l), params, egy, egyd, Te[l], Zed[l], egx, egxd, ez, ezd,
                                      st));
    }
    ProfScope _ps(io.prof, "grad_emb_w", st);
    launch_wgrad<R>(emb_layer(l), emb_shape(l), Ye[l - 1], Yed[l - 1], ez, ezd, emb_ld(l), grad, st);
    std::swap(egy, egx);
    std::swap(egyd, egxd);
  }
  {
    const long rpb = 2048;
    const size_t sm = sizeof(R) * (size_t)m.n_embed_nets * w1 * 2;
    k_emb0_rev<R><<<nb(rows, (int)rpb), 256, sm, st>>>(pc, tsorted, Renv, Rdot, w1, emb_ld(0), egy, egyd, Te[0], Zed[0],
                                                      rpb,
                                                      grad, off);
  }
  DP_CUDA_TRY(cudaGetLastError());
  *grad_out = grad;
  return DP_OK;
}

int run_param_grad(const DeviceModel& m, const PathConst& pc, const PathIO& io, const double* w_dev,
                   const double* a_dev, const double* gv_dev, double b, double* grad, Arena& ar, cudaStream_t st) {
  if (m.compressed || (m.precision != DP_PREC_FP64 && m.precision != DP_PREC_FP32)) {
    set_error("parameter gradients need an uncompressed FP64 or FP32 model");
    return DP_E_UNSUPPORTED;
  }
  if (m.precision == DP_PREC_FP64) {
    double* g = nullptr;
    const int rc = run_grad<double>(m, pc, m.p64, io, w_dev, a_dev, gv_dev, b, ar, st, &g);
    if (rc != DP_OK || ar.measure) return rc;
    DP_CUDA_TRY(cudaMemcpyAsync(grad, g, sizeof(double) * m.n_params, cudaMemcpyDeviceToDevice, st));
    return DP_OK;
  }
  float* g = nullptr;
  const int rc = run_grad<float>(m, pc, m.p32, io, w_dev, a_dev, gv_dev, b, ar, st, &g);
  if (rc != DP_OK || ar.measure) return rc;
  k_to_double<float><<<nb(m.n_params, 256), 256, 0, st>>>(g, m.n_params, grad);
  DP_CUDA_TRY(cudaGetLastError());
  return DP_OK;
}

}  // namespace dpgb
