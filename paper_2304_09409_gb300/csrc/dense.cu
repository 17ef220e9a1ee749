// Dense layer of Eq. (NN) on CUDA cores for FP64 and FP32: forward, input gradient, and (for the
// parameter gradient) forward with tangent and its reverse; dense.cuh gives the formulas.
//
// One launch covers every net of a layer (all type pairs, or all centre types): a block finds the
// net its rows belong to.  Rows are consecutive, or come from a list of the real slot rows (padding
// left out).  A ring of K chunks is filled with cp.async; the tile shape is chosen by the work there
// is (launch_dense).  An FP32 output is one chain of FMAs over k in ascending order whatever the
// shape, so its rounding never depends on the shape; FP64 launches with few tiles split K.
//
// Bounds: FP64 the FP64 pipe (85-95 % busy in every layer of the 192-atom water frame), so columns are
// padded as little as possible and few tiles are split until every SM works: fitting net of that frame
// 7.05 -> 0.58 ms, embedding 2.35 -> 0.77 ms against one 64 x 64 tile per block and a launch per net.
// FP32 latency and instruction issue: 1,029-atom water frame, fitting net 0.81 -> 0.17 ms, embedding
// 0.57 -> 0.20 ms; 6,144-atom training batch, tangent and reverse layers with their tanh passes
// 8.6 -> 2.4 ms.
#include <cooperative_groups.h>

#include <algorithm>
#include <cstring>

#include "dense.cuh"

namespace dpgb {

namespace {

namespace cg = cooperative_groups;

enum DenseMode { DENSE_FWD = 0, DENSE_BWD = 1, DENSE_TAN = 2, DENSE_REV = 3 };
constexpr bool is_fwd(int mode) { return mode == DENSE_FWD || mode == DENSE_TAN; }
// input arrays staged per chunk (X; GY, T; X, Xd; GY, GYd, T, Zd) and accumulator sets
constexpr int n_src(int mode) { return mode == DENSE_FWD ? 1 : mode == DENSE_REV ? 4 : 2; }
constexpr int n_acc(int mode) { return mode == DENSE_TAN || mode == DENSE_REV ? 2 : 1; }

template <class R>
struct DenseJob {
  DenseRows rows;
  int tile0[kMaxDenseGroups];  // first row tile of every group
  int n_in, n_out, skip, act;
  int lda, ldy;    // row strides of the input and output arrays (elements)
  const R* params;
  const R* a[4];   // inputs, in the order of n_src
  R* y[4];         // forward Y, T, (Yd, Zd); reverse GX, (GXd, GZ, GZd)
};

__device__ __forceinline__ double act_tanh(double z) { return tanh(z); }
__device__ __forceinline__ float act_tanh(float z) { return tanhf(z); }

template <class R>
struct __align__(4 * sizeof(R)) Quad {
  R v[4];
};

template <class R>
__device__ __forceinline__ void store_quad(R* p, const R* v, int nv, bool vec) {
  if (vec && nv >= 4) {
    Quad<R> x;
#pragma unroll
    for (int e = 0; e < 4; ++e) x.v[e] = v[e];
    *reinterpret_cast<Quad<R>*>(p) = x;
  } else {
#pragma unroll
    for (int e = 0; e < 4; ++e)
      if (e < nv) p[e] = v[e];
  }
}

// Bias, activation, skip and the stores of four consecutive output columns of one row.
template <class R, int MODE>
__device__ __forceinline__ void epilogue_quad(const DenseJob<R>& g, const R* __restrict__ W, long row, int c,
                                              R acc[n_acc(MODE)][4]) {
  const int n = is_fwd(MODE) ? g.n_out : g.n_in;
  const int nv = n - c;
  if (nv <= 0) return;
  const bool vec = (g.ldy & 3) == 0;
  const long out = row * g.ldy + c;
  if constexpr (is_fwd(MODE)) {
    const R* b = W + (long)g.n_in * g.n_out + c;
    R t[4], y[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const R z = acc[0][e] + (e < nv ? b[e] : R(0));
      t[e] = g.act ? act_tanh(z) : z;
      y[e] = t[e];
    }
    if (g.skip) {
      const R* x = g.a[0] + row * g.lda;
#pragma unroll
      for (int e = 0; e < 4; ++e)
        if (e < nv) y[e] += x[c + e < g.n_in ? c + e : c + e - g.n_in];
    }
    store_quad(g.y[0] + out, y, nv, vec);
    store_quad(g.y[1] + out, t, nv, vec);
    if constexpr (MODE == DENSE_TAN) {
      R yd[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) yd[e] = (R(1) - t[e] * t[e]) * acc[1][e];
      if (g.skip) {
        const R* x = g.a[1] + row * g.lda;
#pragma unroll
        for (int e = 0; e < 4; ++e)
          if (e < nv) yd[e] += x[c + e < g.n_in ? c + e : c + e - g.n_in];
      }
      store_quad(g.y[2] + out, yd, nv, vec);
      store_quad(g.y[3] + out, acc[1], nv, vec);
    }
  } else {
#pragma unroll
    for (int h = 0; h < n_acc(MODE); ++h) {
      if (g.skip) {
        const R* gy = g.a[h] + row * g.lda + c;
#pragma unroll
        for (int e = 0; e < 4; ++e)
          if (e < nv) acc[h][e] += g.skip == 1 ? gy[e] : gy[e] + gy[e + n];
      }
      store_quad(g.y[h] + out, acc[h], nv, vec);
    }
  }
}

// cp.async of BYTES (4, 8 or 16) bytes, the first `valid` of them read and the rest zero-filled.
template <int BYTES>
__device__ __forceinline__ void copy_async(void* dst, const void* src, int valid) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  if constexpr (BYTES == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(valid) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;" ::"r"(d), "l"(src), "n"(BYTES), "r"(valid) : "memory");
}

// Tile geometry shared by the kernels: (BM / TM) x (BN / 4) threads, thread (ty, tx) owns rows
// ty + TY p and four consecutive columns.  A chunks are [row][k] (read as quads along k, broadcast
// across a row's threads), W chunks [k][column].
template <class R, int MODE, int BM, int BN, int TM, int BK>
struct Tile {
  static constexpr int TX = BN / 4, TY = BM / TM, NT = TX * TY;
  static constexpr int LDA = BK + 4, LDB = BN + 4;  // 4-element aligned rows, staggered over the banks
  static constexpr int NSRC = n_src(MODE), NACC = n_acc(MODE);
  static constexpr int RSTEP = NT / (BK / 4), AQ = (BM + RSTEP - 1) / RSTEP;
  static_assert(RSTEP * (BK / 4) == NT, "whole rows of A per pass");
  static constexpr int ASTAGE = NSRC * BM * LDA;

  // copies of this thread's quads of one A chunk: columns k .. k + 3 of rows s_row[ra + q RSTEP]
  static __device__ __forceinline__ void fetch_a(const DenseJob<R>& g, const int* s_row, int ra, int ka, int k, int K,
                                                 R* A) {
    const bool vec = (g.lda & 3) == 0;
#pragma unroll
    for (int q = 0; q < AQ; ++q) {
      const int r = ra + q * RSTEP;
      if (AQ * RSTEP != BM && r >= BM) break;
      const int row = s_row[r];
      const int left = row >= 0 ? K - k : 0;  // real columns from this quad on
      const long at = (long)row * g.lda + k;
#pragma unroll
      for (int h = 0; h < NSRC; ++h) {
        if (MODE == DENSE_BWD && h == 1 && !g.act) continue;
        const R* src = g.a[h] + at;
        R* dst = A + (h * BM + r) * LDA + ka;
        if (vec) {
          constexpr int PER = 16 / sizeof(R);
#pragma unroll
          for (int j = 0; j < 4; j += PER) {
            const int v = min(max(left - j, 0), PER);
            copy_async<16>(dst + j, v ? src + j : g.a[h], v * (int)sizeof(R));
          }
        } else {
#pragma unroll
          for (int j = 0; j < 4; ++j)
            copy_async<sizeof(R)>(dst + j, j < left ? src + j : g.a[h], j < left ? sizeof(R) : 0);
        }
      }
    }
  }
  // GY -> GZ (and the tangent's) on the quads this thread copied; REV: also written out where asked
  static __device__ __forceinline__ void gate_a(const DenseJob<R>& g, const int* s_row, int ra, int ka, int k, int K,
                                                R* A, bool write) {
    if constexpr (MODE == DENSE_BWD) {
      if (!g.act) return;
#pragma unroll
      for (int q = 0; q < AQ; ++q) {
        const int r = ra + q * RSTEP;
        if (AQ * RSTEP != BM && r >= BM) break;
        Quad<R>* y = reinterpret_cast<Quad<R>*>(A + r * LDA + ka);
        const Quad<R> t = *reinterpret_cast<const Quad<R>*>(A + (BM + r) * LDA + ka);
        Quad<R> v = *y;
#pragma unroll
        for (int j = 0; j < 4; ++j) v.v[j] *= R(1) - t.v[j] * t.v[j];
        *y = v;
      }
    } else if constexpr (MODE == DENSE_REV) {
      const bool vec = (g.lda & 3) == 0;
#pragma unroll
      for (int q = 0; q < AQ; ++q) {
        const int r = ra + q * RSTEP;
        if (AQ * RSTEP != BM && r >= BM) break;
        Quad<R>* y = reinterpret_cast<Quad<R>*>(A + r * LDA + ka);
        Quad<R>* yd = reinterpret_cast<Quad<R>*>(A + (BM + r) * LDA + ka);
        const Quad<R> t = *reinterpret_cast<const Quad<R>*>(A + (2 * BM + r) * LDA + ka);
        const Quad<R> zd = *reinterpret_cast<const Quad<R>*>(A + (3 * BM + r) * LDA + ka);
        Quad<R> v = *y, vd = *yd;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const R gate = R(1) - t.v[j] * t.v[j], gyd = vd.v[j];
          vd.v[j] = gyd * gate;
          v.v[j] = (v.v[j] - R(2) * t.v[j] * zd.v[j] * gyd) * gate;
        }
        *y = v;
        *yd = vd;
        const int row = s_row[r];
        if (write && row >= 0) {
          store_quad(g.y[2] + (long)row * g.lda + k, v.v, K - k, vec);
          store_quad(g.y[3] + (long)row * g.lda + k, vd.v, K - k, vec);
        }
      }
    }
  }
  // acc += A chunk x W chunk (k rows of W at B, kn of them real)
  static __device__ __forceinline__ void mma(const R* A, const R* B, int kn, R acc[NACC][TM][4]) {
    auto step = [&](int k4) {
      Quad<R> b[4];
#pragma unroll
      for (int kk = 0; kk < 4; ++kk) b[kk] = *reinterpret_cast<const Quad<R>*>(B + (k4 + kk) * LDB);
#pragma unroll
      for (int h = 0; h < NACC; ++h) {
        Quad<R> a[TM];
#pragma unroll
        for (int p = 0; p < TM; ++p) a[p] = *reinterpret_cast<const Quad<R>*>(A + (h * BM + p * TY) * LDA + k4);
#pragma unroll
        for (int kk = 0; kk < 4; ++kk)
#pragma unroll
          for (int p = 0; p < TM; ++p)
#pragma unroll
            for (int q = 0; q < 4; ++q) acc[h][p][q] += a[p].v[kk] * b[kk].v[q];
      }
    };
    if (kn >= BK) {
#pragma unroll
      for (int k4 = 0; k4 < BK; k4 += 4) step(k4);
    } else {  // the last chunk: no work beyond K (rounded up to 4)
#pragma unroll 1
      for (int k4 = 0; k4 < kn; k4 += 4) step(k4);
    }
  }
};

// One output tile per block.  SPLIT (FP64): the blocks of a cluster take consecutive parts of K, their
// partial tiles meet through distributed shared memory in a fixed order and each block finishes
// BM / cluster rows.
template <class R, int MODE, int BM, int BN, int TM, int BK, int ST, bool SPLIT>
__global__ void __launch_bounds__((BM / TM) * (BN / 4))
    k_dense(const __grid_constant__ DenseJob<R> g) {
  using T = Tile<R, MODE, BM, BN, TM, BK>;
  constexpr int TX = T::TX, TY = T::TY, NT = T::NT, LDA = T::LDA, LDB = T::LDB, NACC = T::NACC;
  constexpr int BE = BN * BK / NT;
  static_assert(BE * NT == BN * BK, "whole passes over the W chunk");
  constexpr int STAGE = T::ASTAGE + BK * LDB;
  extern __shared__ __align__(32) unsigned char smem_raw[];
  R* smem = reinterpret_cast<R*>(smem_raw);  // [ST][A arrays | W]
  __shared__ int s_row[BM];

  const int tid = threadIdx.x, tx = tid % TX, ty = tid / TX;
  const int cs = SPLIT ? (int)gridDim.x : 1;  // the blocks along x form one cluster over K
  const int cr = SPLIT ? (int)blockIdx.x : 0;
  const int tile = SPLIT ? (int)blockIdx.z : (int)blockIdx.x;
  const int c0 = (int)blockIdx.y * BN;
  int gi = 0;
  while (gi + 1 < g.rows.ngroups && tile >= g.tile0[gi + 1]) ++gi;
  const DenseGroup grp = g.rows.g[gi];
  const int nrows = g.rows.rows_of(gi);
  const int r0 = (tile - g.tile0[gi]) * BM;
  if (r0 >= nrows) return;  // the whole cluster leaves: the rows do not depend on cr
  for (int r = tid; r < BM; r += NT) {
    int row = -1;
    if (r0 + r < nrows) row = g.rows.list ? __ldg(g.rows.list + grp.r0 + r0 + r) : (int)grp.r0 + r0 + r;
    s_row[r] = row;
  }
  __syncthreads();

  const R* __restrict__ W = g.params + grp.w;
  const int K = is_fwd(MODE) ? g.n_in : g.n_out;
  const int N = is_fwd(MODE) ? g.n_out : g.n_in;
  const int nch = (K + BK - 1) / BK;
  const int ch0 = (int)((long)nch * cr / cs), ch1 = (int)((long)nch * (cr + 1) / cs);
  const int ra = tid / (BK / 4), ka = 4 * (tid % (BK / 4));
  // W chunk: element (kb + q KSTEP, cb) forward (lanes along the columns of W), (kb, cb + q CSTEP)
  // for W^T (lanes along the rows of W, i.e. along k); chunks come in order, so the address advances
  constexpr int KSTEP = is_fwd(MODE) ? NT / BN : 0, CSTEP = is_fwd(MODE) ? 0 : NT / BK;
  static_assert(is_fwd(MODE) ? NT % BN == 0 : NT % BK == 0, "W elements in whole rows per pass");
  const int kb = is_fwd(MODE) ? tid / BN : tid % BK, cb = is_fwd(MODE) ? tid % BN : tid / BK;
  int bk = ch0 * BK + kb, ak = ch0 * BK + ka;
  const R* pb = is_fwd(MODE) ? W + (long)bk * g.n_out + c0 + cb : W + (long)(c0 + cb) * g.n_out + bk;
  const long bq = (long)(is_fwd(MODE) ? KSTEP : CSTEP) * g.n_out;
  const long bch = is_fwd(MODE) ? (long)BK * g.n_out : BK;
  int fst = 0;  // stage of the next fetch
  auto fetch = [&]() {
    R* A = smem + fst * STAGE;
    T::fetch_a(g, s_row, ra, ka, ak, K, A);
    R* B = A + T::ASTAGE + kb * LDB + cb;
#pragma unroll
    for (int q = 0; q < BE; ++q) {
      const bool on = bk + q * KSTEP < K && c0 + cb + q * CSTEP < N;
      copy_async<sizeof(R)>(B + q * KSTEP * LDB + q * CSTEP, on ? pb + q * bq : W, on ? sizeof(R) : 0);
    }
    ak += BK;
    bk += BK;
    pb += bch;
    fst = fst + 1 == ST ? 0 : fst + 1;
  };
  R acc[NACC][TM][4];
#pragma unroll
  for (int h = 0; h < NACC; ++h)
#pragma unroll
    for (int p = 0; p < TM; ++p)
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[h][p][q] = R(0);
#pragma unroll
  for (int s = 0; s < ST - 1; ++s) {
    if (ch0 + s < ch1) fetch();
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  int cst = 0;  // stage of chunk ch
  for (int ch = ch0; ch < ch1; ++ch) {
    asm volatile("cp.async.wait_group %0;" ::"n"(ST - 2) : "memory");  // this thread's part of chunk ch
    R* A = smem + cst * STAGE;
    cst = cst + 1 == ST ? 0 : cst + 1;
    T::gate_a(g, s_row, ra, ka, ch * BK + ka, K, A, blockIdx.y == 0);
    __syncthreads();  // chunk ch is complete, and every thread is done with chunk ch - 1
    if (ch + ST - 1 < ch1) fetch();
    asm volatile("cp.async.commit_group;" ::: "memory");
    T::mma(A + ty * LDA, A + T::ASTAGE + tx * 4, K - ch * BK, acc);
  }
  if (SPLIT && cs > 1) {
    cg::cluster_group cluster = cg::this_cluster();
    __syncthreads();  // the ring is no longer read
    R* part = smem;   // [NACC][BM][BN]
#pragma unroll
    for (int h = 0; h < NACC; ++h)
#pragma unroll
      for (int p = 0; p < TM; ++p) {
        Quad<R> x;
#pragma unroll
        for (int q = 0; q < 4; ++q) x.v[q] = acc[h][p][q];
        *reinterpret_cast<Quad<R>*>(part + (h * BM + ty + TY * p) * BN + tx * 4) = x;
      }
    cluster.sync();
    const int rows_each = BM / cs;
    for (int e = tid; e < rows_each * TX; e += NT) {
      const int r = cr * rows_each + e / TX, c = (e % TX) * 4;
      if (s_row[r] < 0) continue;
      R v[NACC][4] = {};
      for (int k = 0; k < cs; ++k)
#pragma unroll
        for (int h = 0; h < NACC; ++h) {
          const Quad<R> x = *reinterpret_cast<const Quad<R>*>(cluster.map_shared_rank(part, k) + (h * BM + r) * BN + c);
#pragma unroll
          for (int j = 0; j < 4; ++j) v[h][j] += x.v[j];
        }
      epilogue_quad<R, MODE>(g, W, s_row[r], c0 + c, v);
    }
    cluster.sync();  // a block's partial tile is read by the others until here
  } else {
#pragma unroll
    for (int p = 0; p < TM; ++p) {
      const int row = s_row[ty + TY * p];
      R v[NACC][4];
#pragma unroll
      for (int h = 0; h < NACC; ++h)
#pragma unroll
        for (int q = 0; q < 4; ++q) v[h][q] = acc[h][p][q];
      if (row >= 0) epilogue_quad<R, MODE>(g, W, row, c0 + tx * 4, v);
    }
  }
}

// Narrow layers over many rows (the embedding nets): K is short, so a tile per block would spend its
// time filling and draining (526k rows, 25 -> 50 -> 100: 492 us with a block per tile, 426 us here).  Persistent blocks take consecutive row tiles, keep the whole W (all N
// columns, N <= BN) in shared memory, and run one ring of A chunks across their tiles: the next tile's
// copies are in flight while this tile's epilogue runs.
template <class R, int MODE, int BM, int BN, int TM, int BK, int ST>
__global__ void __launch_bounds__((BM / TM) * (BN / 4))
    k_dense_rows(const __grid_constant__ DenseJob<R> g) {
  using T = Tile<R, MODE, BM, BN, TM, BK>;
  constexpr int TX = T::TX, TY = T::TY, NT = T::NT, LDA = T::LDA, LDB = T::LDB, NACC = T::NACC;
  // rows of a tile are in their slot kAhead tiles ahead, and on their way from memory one more
  constexpr int kAhead = ST - 1, kSlots = kAhead + 2;
  static_assert(BM <= NT, "one row look-up per thread");
  extern __shared__ __align__(32) unsigned char smem_raw[];
  R* ring = reinterpret_cast<R*>(smem_raw);      // [ST][A arrays]
  R* Ws = ring + ST * T::ASTAGE;                 // [K rounded up to 4][LDB]
  __shared__ int s_row[kSlots][BM];
  __shared__ int s_tile0[kMaxDenseGroups + 1];

  const int tid = threadIdx.x, tx = tid % TX, ty = tid / TX;
  const int K = is_fwd(MODE) ? g.n_in : g.n_out;
  const int N = is_fwd(MODE) ? g.n_out : g.n_in;
  const int ng = g.rows.ngroups;
  if (tid == 0) {  // row tiles of the rows there really are
    int at = 0;
    for (int k = 0; k < ng; ++k) {
      s_tile0[k] = at;
      at += (g.rows.rows_of(k) + BM - 1) / BM;
    }
    s_tile0[ng] = at;
  }
  __syncthreads();
  const int total = s_tile0[ng];
  const int t0 = (int)((long)total * blockIdx.x / gridDim.x), t1 = (int)((long)total * (blockIdx.x + 1) / gridDim.x);
  if (t0 >= t1) return;
  auto group_of = [&](int tile) {
    int k = 0;
    while (k + 1 < ng && tile >= s_tile0[k + 1]) ++k;
    return k;
  };
  auto look_up = [&](int tile) {  // thread r: row r of the tile (-1 beyond its end)
    if (tid >= BM || tile >= t1) return -1;
    const int k = group_of(tile);
    const DenseGroup& grp = g.rows.g[k];
    const int nrows = g.rows.rows_of(k);
    const int r = (tile - s_tile0[k]) * BM + tid;
    if (r >= nrows) return -1;
    return g.rows.list ? __ldg(g.rows.list + grp.r0 + r) : (int)grp.r0 + r;
  };
  for (int a = 0; a < kAhead; ++a)
    if (tid < BM) s_row[a][tid] = look_up(t0 + a);
  int ahead = look_up(t0 + kAhead);
  __syncthreads();
  const int nch = (K + BK - 1) / BK;
  const int ra = tid / (BK / 4), ka = 4 * (tid % (BK / 4));
  int ft = t0, fch = 0, fst = 0;  // tile, chunk and stage of the next fetch
  auto fetch = [&]() {
    if (ft < t1) {
      T::fetch_a(g, s_row[(ft - t0) % kSlots], ra, ka, fch * BK + ka, K, ring + fst * T::ASTAGE);
      if (++fch == nch) {
        fch = 0;
        ++ft;
      }
      fst = fst + 1 == ST ? 0 : fst + 1;
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
#pragma unroll
  for (int s = 0; s < ST - 1; ++s) fetch();
  int cur = -1, cst = 0;
  const R* W = nullptr;
  for (int tile = t0; tile < t1; ++tile) {
    const int k = group_of(tile);
    if (k != cur) {  // the net of the rows changes (block-uniform)
      cur = k;
      W = g.params + g.rows.g[k].w;
      __syncthreads();  // the previous net's W is no longer read
      const int kp = (K + 3) & ~3;
      for (int e = tid; e < kp * BN; e += NT) {
        // lanes along the contiguous direction of W
        const int kk = is_fwd(MODE) ? e / BN : e % kp, c = is_fwd(MODE) ? e % BN : e / kp;
        Ws[kk * LDB + c] =
            kk < K && c < N ? __ldg(W + (is_fwd(MODE) ? (long)kk * g.n_out + c : (long)c * g.n_out + kk)) : R(0);
      }
    }
    const int* rows = s_row[(tile - t0) % kSlots];
    R acc[NACC][TM][4];
#pragma unroll
    for (int h = 0; h < NACC; ++h)
#pragma unroll
      for (int p = 0; p < TM; ++p)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[h][p][q] = R(0);
    for (int ch = 0; ch < nch; ++ch) {
      asm volatile("cp.async.wait_group %0;" ::"n"(ST - 2) : "memory");
      R* A = ring + cst * T::ASTAGE;
      cst = cst + 1 == ST ? 0 : cst + 1;
      T::gate_a(g, rows, ra, ka, ch * BK + ka, K, A, true);
      if (ch == 0) {  // the slot was last read by the epilogue of tile - 2
        if (tid < BM) s_row[(tile - t0 + kAhead) % kSlots][tid] = ahead;
        ahead = look_up(tile + kAhead + 1);
      }
      __syncthreads();  // the chunk (and W, and the looked-up rows) are complete; the last chunk was read
      fetch();
      T::mma(A + ty * LDA, Ws + ch * BK * LDB + tx * 4, K - ch * BK, acc);
    }
#pragma unroll
    for (int p = 0; p < TM; ++p) {
      const int row = rows[ty + TY * p];
      R v[NACC][4];
#pragma unroll
      for (int h = 0; h < NACC; ++h)
#pragma unroll
        for (int q = 0; q < 4; ++q) v[h][q] = acc[h][p][q];
      if (row >= 0) epilogue_quad<R, MODE>(g, W, row, tx * 4, v);
    }
  }
}

template <class R, int MODE, int BM, int BN, int TM, int BK, int ST, bool SPLIT>
cudaError_t launch_shape(DenseJob<R>& g, int cs, cudaStream_t st) {
  using T = Tile<R, MODE, BM, BN, TM, BK>;
  int tiles = 0;
  for (int k = 0; k < g.rows.ngroups; ++k) {
    g.tile0[k] = tiles;
    tiles += (g.rows.g[k].nrows + BM - 1) / BM;
  }
  const int N = is_fwd(MODE) ? g.n_out : g.n_in;
  constexpr size_t stages = sizeof(R) * ST * (T::ASTAGE + BK * T::LDB);
  constexpr size_t part = SPLIT ? sizeof(R) * T::NACC * BM * BN : 0;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = SPLIT ? dim3(cs, (N + BN - 1) / BN, tiles) : dim3(tiles, (N + BN - 1) / BN, 1);
  cfg.blockDim = dim3(T::NT);
  cfg.dynamicSmemBytes = stages > part ? stages : part;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = cs;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = SPLIT && cs > 1 ? 1 : 0;
  auto kernel = k_dense<R, MODE, BM, BN, TM, BK, ST, SPLIT>;
  if (cfg.dynamicSmemBytes > 47 * 1024) {
    const cudaError_t e = allow_max_smem(kernel);
    if (e != cudaSuccess) return e;
  }
  return cudaLaunchKernelEx(&cfg, kernel, g);
}

template <class R, int MODE, int BM, int BN, int TM, int BK, int ST>
cudaError_t launch_rows(DenseJob<R>& g, cudaStream_t st) {
  using T = Tile<R, MODE, BM, BN, TM, BK>;
  const int K = is_fwd(MODE) ? g.n_in : g.n_out;
  const size_t smem = sizeof(R) * (size_t)(ST * T::ASTAGE + ((K + 3) & ~3) * T::LDB);
  auto kernel = k_dense_rows<R, MODE, BM, BN, TM, BK, ST>;
  cudaError_t e = allow_max_smem(kernel);
  int per_sm = 1;
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, T::NT, smem);
  if (e != cudaSuccess) return e;
  kernel<<<sm_count() * std::max(1, per_sm), T::NT, smem, st>>>(g);
  return cudaGetLastError();
}

template <class R, int MODE>
cudaError_t launch_dense(DenseJob<R>& g, cudaStream_t st) {
  const int N = is_fwd(MODE) ? g.n_out : g.n_in, K = is_fwd(MODE) ? g.n_in : g.n_out;
  constexpr bool DUAL = n_acc(MODE) == 2;
  long rows = 0, t32 = 0, t64 = 0, t128 = 0;
  for (int k = 0; k < g.rows.ngroups; ++k) {
    const long n = g.rows.g[k].nrows;
    rows += n;
    t32 += (n + 31) / 32;
    t64 += (n + 63) / 64;
    t128 += (n + 127) / 128;
  }
  if (rows == 0) return cudaSuccess;
  const long sms = sm_count();
  // column tile: the one of 64, 52, 32 that pads N least (100 = 2 x 52, 50 -> 52, 25 -> 32)
  int bn = 64;
  auto padded = [&](int w) { return (N + w - 1) / w * w; };
  if (padded(52) < padded(bn)) bn = 52;
  if (padded(32) < padded(bn)) bn = 32;
  const long nbn = padded(bn) / bn, n32 = (N + 31) / 32;
  // 64-row tiles once they give every SM four blocks; the split 32 x 32 ones below that (64 x 64 tiles put
  // the 192-atom frame's first fitting layer on 12 SMs: 2.7 ms against 0.21 ms)
  if constexpr (sizeof(R) == 8) {
    if (t64 * nbn >= 4 * sms) {
      if (bn == 32) return launch_shape<R, MODE, 64, 32, 2, 16, 2, false>(g, 1, st);
      if (bn == 52) return launch_shape<R, MODE, 64, 52, 4, 16, 2, false>(g, 1, st);
      return launch_shape<R, MODE, 64, 64, 4, 16, 2, false>(g, 1, st);
    }
    // blocks along K: as many (1, 2, 4, 8) as keep two chunks of K for every block and the grid within
    // two blocks a SM
    int cs = 1;
    while (cs < 8 && t32 * n32 * cs * 2 <= 2 * sms && (K + 15) / 16 >= 4 * cs) cs *= 2;
    return launch_shape<R, MODE, 32, 32, 2, 16, 3, true>(g, cs, st);
  } else {
    if (K <= 128 && N <= 128 && t64 >= 4 * sms) {
      constexpr int TM = DUAL ? 4 : 8;            // rows a thread of the widest tiles
      constexpr int ST = MODE == DENSE_REV ? 2 : 3;  // four arrays a chunk: two stages keep three blocks a SM
      if (N <= 32) return launch_rows<R, MODE, 64, 32, 2, 16, ST>(g, st);
      if (N <= 52) return launch_rows<R, MODE, 64, 52, 4, 16, ST>(g, st);
      if (N <= 64) return launch_rows<R, MODE, 64, 64, 4, 16, ST>(g, st);
      if (N <= 104) return launch_rows<R, MODE, 8 * TM, 104, TM, 16, ST>(g, st);
      return launch_rows<R, MODE, 8 * TM, 128, TM, 16, ST>(g, st);
    }
    // 128-row tiles once every SM has four of them, 64-row ones while every SM has one (4,116 atoms,
    // 1,640 -> 240: 107 us against 150 us in 32 x 32 tiles), else 32 x 32 tiles for the number of blocks
    if constexpr (!DUAL) {
      if (t128 * nbn >= 4 * sms) {
        if (bn == 32) return launch_shape<R, MODE, 128, 32, 4, 16, 3, false>(g, 1, st);
        if (bn == 52) return launch_shape<R, MODE, 128, 52, 8, 16, 3, false>(g, 1, st);
        return launch_shape<R, MODE, 128, 64, 8, 16, 3, false>(g, 1, st);
      }
    }
    if (bn > 32 && t64 * nbn >= sms) {
      if (bn == 52) return launch_shape<R, MODE, 64, 52, 4, 16, 3, false>(g, 1, st);
      return launch_shape<R, MODE, 64, 64, 4, 16, 3, false>(g, 1, st);
    }
    return launch_shape<R, MODE, 32, 32, 2, 32, DUAL ? 3 : 4, false>(g, 1, st);
  }
}

template <class R>
DenseJob<R> make_job(const DenseRows& rows, const DenseShape& s, bool fwd, const R* params) {
  DenseJob<R> g;
  std::memset(&g, 0, sizeof(g));
  g.rows = rows;
  g.n_in = s.n_in;
  g.n_out = s.n_out;
  g.skip = s.skip;
  g.act = s.act;
  g.lda = fwd ? s.ldx : s.ldy;
  g.ldy = fwd ? s.ldy : s.ldx;
  g.params = params;
  return g;
}

}  // namespace

template <class R>
cudaError_t launch_dense_fwd(const DenseRows& rows, const DenseShape& s, const R* params, const R* X, R* Y, R* T,
                             cudaStream_t st) {
  DenseJob<R> g = make_job<R>(rows, s, true, params);
  g.a[0] = X;
  g.y[0] = Y;
  g.y[1] = T;
  return launch_dense<R, DENSE_FWD>(g, st);
}

template <class R>
cudaError_t launch_dense_bwd(const DenseRows& rows, const DenseShape& s, const R* params, const R* GY, const R* T,
                             R* GX, cudaStream_t st) {
  DenseJob<R> g = make_job<R>(rows, s, false, params);
  g.a[0] = GY;
  g.a[1] = T;
  g.y[0] = GX;
  return launch_dense<R, DENSE_BWD>(g, st);
}

template <class R>
cudaError_t launch_dense_tan(const DenseRows& rows, const DenseShape& s, const R* params, const R* X, const R* Xd,
                             R* Y, R* T, R* Yd, R* Zd, cudaStream_t st) {
  DenseJob<R> g = make_job<R>(rows, s, true, params);
  g.a[0] = X;
  g.a[1] = Xd;
  g.y[0] = Y;
  g.y[1] = T;
  g.y[2] = Yd;
  g.y[3] = Zd;
  return launch_dense<R, DENSE_TAN>(g, st);
}

template <class R>
cudaError_t launch_dense_rev(const DenseRows& rows, const DenseShape& s, const R* params, const R* GY, const R* GYd,
                             const R* T, const R* Zd, R* GX, R* GXd, R* GZ, R* GZd, cudaStream_t st) {
  DenseJob<R> g = make_job<R>(rows, s, false, params);
  g.a[0] = GY;
  g.a[1] = GYd;
  g.a[2] = T;
  g.a[3] = Zd;
  g.y[0] = GX;
  g.y[1] = GXd;
  g.y[2] = GZ;
  g.y[3] = GZd;
  return launch_dense<R, DENSE_REV>(g, st);
}

#define DPGB_DENSE(R)                                                                                                \
  template cudaError_t launch_dense_fwd<R>(const DenseRows&, const DenseShape&, const R*, const R*, R*, R*,          \
                                           cudaStream_t);                                                            \
  template cudaError_t launch_dense_bwd<R>(const DenseRows&, const DenseShape&, const R*, const R*, const R*, R*,    \
                                           cudaStream_t);                                                            \
  template cudaError_t launch_dense_tan<R>(const DenseRows&, const DenseShape&, const R*, const R*, const R*, R*,    \
                                           R*, R*, R*, cudaStream_t);                                                \
  template cudaError_t launch_dense_rev<R>(const DenseRows&, const DenseShape&, const R*, const R*, const R*,        \
                                           const R*, const R*, R*, R*, R*, R*, cudaStream_t);
DPGB_DENSE(double)
DPGB_DENSE(float)
#undef DPGB_DENSE

}  // namespace dpgb
