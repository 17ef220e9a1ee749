// The whole fitting net of the FP32 mode -- forward to E_i and backward to dE/dD -- in one tcgen05
// kernel per 128-atom tile, on split BF16 operands (x = hi + lo, every product formed as
// hi.hi + hi.lo + lo.hi: about 16 significant bits per operand, FP32 accumulation), Eq.
// (fitting_energy) with the layers of Eq. (NN).
//
// Per tile the CTA runs the chain of GEMMs of the net: forward layers z_l = y_{l-1} W_l + b_l,
// t_l = tanh z_l, y_l = t_l (+ y_{l-1}), E = y_last . w + b; backward gz_last = w (1 - t_last^2),
// gy_{l-1} = gz_l W_l^T (+ gy_l), gz_{l-1} = gy_{l-1} (1 - t_{l-1}^2), dE/dD = gz_0 W_0^T.
//
// What bounds it is the chain: one tile per SM, every phase's MMAs (2.9 us at K = 240) and the epilogue
// between two phases (7-9 us) follow each other.  So nothing else may stand in that chain:
//   - the activations stay in shared memory: an epilogue writes the next phase's A operand, high and low
//     BF16 halves in the tensor core's 128-byte-swizzled layout, 64 columns at a time, and the next
//     phase's MMAs start on each 64-column block as soon as it is written (two accumulators in tensor
//     memory, phases alternate);
//   - weights come through a ring of their own, 32 columns of K a slot (64-byte swizzle; 64 columns of
//     high and low halves for 240 outputs would not fit twice beside the operand), filled during the
//     epilogue before;
//   - the descriptor of the first phase streams through four stages over the whole buffer, which the
//     operand and the ring then take over;
//   - the FP32 residual stream (y_l, gy_l) and the gates 1 - t^2 go to an L2-resident scratch that the
//     thread that wrote them reads back.
// dE/dD leaves in 192-column chunks from two accumulators, so that a chunk's epilogue overlaps the next
// one's MMAs.  To have two of 192 columns in tensor memory and five weight slots in shared memory, the
// chunks' operand gz_0 is split: its high half goes to tensor memory (the MMA reads A from there), its low
// half to shared memory.  With M_< = 16 each 16-column piece is one m of dE/dD[m][l] and is folded into
// dE/dT at once, T_< of a thread's row in registers.
// One tile on 12,288 water atoms, thousand clocks (first GEMM; five epilogues; the four GEMMs between them;
// chunks; end): 56; 85; 43; 86; 11 (147 us) when each epilogue stored its operand to L2 for the next phase
// to load, now 47; 64; 22; 66; 3 (107 us).  The first GEMM is at the shared memory's bandwidth, the
// epilogues at about half their instruction issue.
// One thread issues TMA, one issues tcgen05.mma, eight warps run the epilogues; every mbarrier wait is
// bounded (on time-out the CTA records an error and finishes).
#include <cuda_bf16.h>

#include <algorithm>
#include <cstring>

#include "fit_tc.cuh"
#include "tc_gemm.cuh"
#include "tc_ptx.cuh"

namespace dpgb {

namespace {

using namespace ptx;

constexpr int kSL = 4;  // hidden layers at most
constexpr int kSEpi = 256;               // eight epilogue warps: two per 32-row quarter of the tile
constexpr int kSThreads = kSEpi + 64;    // + a TMA producer warp and an MMA warp
constexpr int kProd = kSEpi / 32, kMmaW = kProd + 1;  // their warp indices
constexpr int kParts = kSEpi / 128;      // epilogue warps sharing a row quarter, interleaved by 16 columns
constexpr int kStep = 16 * kParts;       // column stride of one epilogue thread
constexpr int SBM = 128;
constexpr int kKB = 32;                   // K columns of one weight slot (64 bytes a row)
constexpr uint32_t kOpBlock = SBM * 128;  // 16 KB: 64 columns of one half of the operand
constexpr uint32_t kOpBytes = 8 * kOpBlock;  // operand: four blocks of the high half, four of the low half
constexpr uint32_t kDHalf = SBM * kKB * 2;   // 8 KB: 32 descriptor columns of one half
constexpr int kP0 = 4;                    // stages of the first phase
constexpr int CH = 192;                   // dE/dD chunk width
constexpr uint32_t kCHalf = CH * kKB * 2; // 12 KB: 32 columns of K of a chunk's weights, one half
constexpr int kCRing = 5;                 // chunk weight slots (high and low half each)
// two slots over the high half of the chain's operand, three behind the low half
__host__ __device__ constexpr uint32_t chunk_slot(int s) {
  return (s < 2 ? 0u : kOpBytes - 2u * 2u * kCHalf) + (uint32_t)s * 2u * kCHalf;
}
constexpr int kSLd = 256;  // row pitch of the residual and gate scratch (elements)

// Weight rows of a chain slot (the widest layer) and ring slots; chunk slots that fit.
__host__ __device__ constexpr int slot_rows(int maxw) { return maxw <= 240 ? 240 : 256; }
__host__ __device__ constexpr int ring_slots(int rows) { return rows == 240 ? 3 : 2; }
__host__ __device__ constexpr int chunk_slots(int rows) { return rows == 240 ? kCRing : kCRing - 1; }
__host__ __device__ constexpr uint32_t slot_bytes(int rows) { return 2u * (uint32_t)rows * kKB * 2u; }
__host__ __device__ constexpr uint32_t buffer_bytes(int rows) {
  return kOpBytes + (uint32_t)ring_slots(rows) * slot_bytes(rows);
}
static_assert(chunk_slot(1) + 2 * kCHalf <= kOpBytes / 2, "two chunk slots fit the operand's high half");
static_assert(chunk_slot(chunk_slots(240)) <= buffer_bytes(240) && chunk_slot(chunk_slots(256)) <= buffer_bytes(256),
              "chunk slots fit");
static_assert(kP0 * (2 * kDHalf + slot_bytes(240)) <= buffer_bytes(240), "first-phase stages fit the buffer");
static_assert(kP0 * (2 * kDHalf + slot_bytes(256)) <= buffer_bytes(256), "first-phase stages fit the buffer");

struct SplitMaps {
  CUtensorMap d[2];                         // D hi / lo [rows][KD], box {32, 128}
  // per type, hi / lo: forward W_l^T (slot l), backward W_l (slot nh + l, l >= 1), box {32, outputs}; W_0 for
  // the chunks (slot nh), box {32, 192}
  CUtensorMap w[DP_MAX_TYPES][2 * kSL][2];
};

struct SplitArgs {
  int ntypes, nh, rows;  // rows of a weight slot
  int width[kSL + 1];  // width[0] = KD, width[l + 1] = outputs of hidden layer l
  int skip[kSL];
  int row_start[DP_MAX_TYPES + 1];
  int tile_start[DP_MAX_TYPES + 1];
  const float* bias[DP_MAX_TYPES][kSL];
  const float* w_last[DP_MAX_TYPES];
  float b_last[DP_MAX_TYPES];
  // scratch of every tile, each value read back by the thread that wrote it: 8-column groups, a row's
  // eight values in one 32-byte sector and the rows of a group contiguous (a warp's access covers 8 lines;
  // with a row pitch of 256 columns it covered 32, and the L1 tag rate bound the epilogues)
  float* resid;             // y_l forward, gy_l backward [tiles][32][128][8]
  float* gate;              // 1 - t_l^2 of the inner hidden layers [nh][tiles][32][128][8]
  const int* perm;
  double* atom_e;
  float* gD;                // dE/dD FP32 [rows][KD], or null when gT is formed instead
  // dE/dT of the se_e2_a contraction (M_< = 16), formed from each dE/dD chunk in the epilogue:
  // gT[m][c] = sum_l gD[m][l] T[l][c] + [m < 16] sum_q gD[q][m] T[q][c], stored m-major
  // [M][rows][4] FP32 (consecutive rows of one m are contiguous)
  float* gT;
  const float* Tm;          // T [rows][M][4] FP32
  int M;
  int* err;
};

// 32-byte global accesses (one full sector per lane): half the instructions and no partial-sector
// writes where each lane owns a row of the tile.
__device__ __forceinline__ void st_v8(float* p, const float* v) {
  asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "f"(v[0]), "f"(v[1]), "f"(v[2]),
               "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7])
               : "memory");
}
__device__ __forceinline__ void ld_v8(const float* p, float* v) {
  asm volatile("ld.global.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7])
               : "l"(p));
}

// tanh from the exponential, tanh x = 1 - 2 / (1 + e^{2x}) (x clamped to +-15, where tanh is 1 to
// FP32): absolute error a few 1e-7, below the ~2^-17 relative rounding the next GEMM's split
// operands apply anyway.  Only the exponential goes to the special-function unit, the epilogues'
// narrowest pipe: 1/d comes from the bit pattern of d (first guess within 5.1 %, the constant
// fitted to the mantissa range [1, 2)) and three Newton steps y <- y (2 - d y) on the FMA pipe.
__device__ __forceinline__ float tanh_ex(float x) {
  const float e = __expf(2.f * fminf(fmaxf(x, -15.f), 15.f));
  const float d = 1.f + e;  // [1, 1 + e^30]: a normal number
  float y = __int_as_float(0x7EF311C0 - __float_as_int(d));
  y = y * (2.f - d * y);
  y = y * (2.f - d * y);
  y = y * (2.f - d * y);
  return 1.f - 2.f * y;
}

__device__ __forceinline__ void split2(float x, __nv_bfloat16& hi, __nv_bfloat16& lo) {
  hi = __float2bfloat16_rn(x);
  lo = __float2bfloat16_rn(x - __bfloat162float(hi));
}

__global__ void __launch_bounds__(kSThreads, 1) k_fit_split(const __grid_constant__ SplitMaps mp, const SplitArgs g) {
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem =
      reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  const uint32_t slotb = slot_bytes(g.rows), halfb = slotb / 2;
  const int NS = ring_slots(g.rows);
  unsigned char* ring = smem + kOpBytes;
  uint64_t* full0 = reinterpret_cast<uint64_t*>(smem + buffer_bytes(g.rows));
  uint64_t* empty0 = full0 + kP0;
  uint64_t* fullw = empty0 + kP0;   // [3]
  uint64_t* emptyw = fullw + 3;     // [3]
  uint64_t* accf = emptyw + 3;      // [2] accumulator ready (MMA -> epilogue)
  uint64_t* accfree = accf + 2;     // [2] dE/dD chunk read (epilogue -> MMA)
  uint64_t* aready = accfree + 2;   // [4] 64-column block of the next operand written (epilogue -> MMA)
  uint64_t* chain_done = aready + 4;  // every MMA of the chain phases has completed
  uint64_t* fullc = chain_done + 1;   // [kCRing]
  uint64_t* emptyc = fullc + kCRing;  // [kCRing]
  uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(emptyc + kCRing + 1);
  float* s_e = reinterpret_cast<float*>(tmem_holder + 4);  // [kParts][128]
  float* s_bias = s_e + kParts * SBM;                      // [kSL][256] biases of the hidden layers
  float* s_wl = s_bias + kSL * 256;                        // [256] weights of the output layer

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int t = 0;
  while (t + 1 < g.ntypes && (int)blockIdx.x >= g.tile_start[t + 1]) ++t;
  const int row0 = g.row_start[t] + ((int)blockIdx.x - g.tile_start[t]) * SBM;
  const int row_end = g.row_start[t + 1];
  const long rows = g.row_start[g.ntypes];
  const int nh = g.nh, KD = g.width[0];
  const int nch = (KD + CH - 1) / CH;
  // chain phases: forward layers 0 .. nh-1, backward layers nh-1 .. 1; phase p accumulates in tensor-memory
  // columns [256 (p & 1), ..).  The last one is even; its epilogue puts the high half of the chunks' operand
  // into columns [384, 512), and chunk c accumulates in columns [192 (c & 1), ..).
  const int nchain = 2 * nh - 1;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kP0; ++s) {
      mbar_init(&full0[s], 1);
      mbar_init(&empty0[s], 1);
    }
    for (int s = 0; s < 3; ++s) {
      mbar_init(&fullw[s], 1);
      mbar_init(&emptyw[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&accf[b], 1);
      mbar_init(&accfree[b], kSEpi);
    }
    for (int b = 0; b < 4; ++b) mbar_init(&aready[b], kSEpi);
    mbar_init(chain_done, 1);
    for (int s = 0; s < kCRing; ++s) {
      mbar_init(&fullc[s], 1);
      mbar_init(&emptyc[s], 1);
    }
    mbar_fence_init();
  }
  if (warp == kProd) tmem_alloc(tmem_holder, 512);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_holder;

  // chain phase p >= 1: its GEMM (K, N) and weight map
  auto phase_info = [&](int p, int& K, int& N, int& wslot) {
    if (p < nh) {
      K = g.width[p];
      N = g.width[p + 1];
      wslot = p;
    } else {  // backward layer l = nh - 1 - (p - nh): A = gz_l
      const int l = nh - 1 - (p - nh);
      K = g.width[l + 1];
      N = g.width[l];
      wslot = nh + l;
    }
  };
  const int nkc = (g.width[1] + kKB - 1) / kKB;  // weight slots' worth of a chunk
  const int NC = chunk_slots(g.rows);
  const uint32_t p0_stage = 2 * kDHalf + slotb;
  const int nk0 = (KD + kKB - 1) / kKB;

  if (warp == kProd) {
    if (lane == 0) {
      // ---- TMA producer ----
      bool ok = true;
      int n0 = 0, it = 0;  // loads issued: first phase, weight ring
      for (int kb = 0; kb < nk0; ++kb) {
        const int s = kb % kP0;
        if (kb >= kP0 && !mbar_wait(&empty0[s], ((kb / kP0) - 1) & 1, g.err)) {
          ok = false;
          break;
        }
        unsigned char* st = smem + s * p0_stage;
        mbar_expect_tx(&full0[s], 2 * kDHalf + 2u * (uint32_t)g.width[1] * kKB * 2u);
        tma_load_2d(st, &mp.d[0], &full0[s], kb * kKB, row0);
        tma_load_2d(st + kDHalf, &mp.d[1], &full0[s], kb * kKB, row0);
        tma_load_2d(st + 2 * kDHalf, &mp.w[t][0][0], &full0[s], kb * kKB, 0);
        tma_load_2d(st + 2 * kDHalf + halfb, &mp.w[t][0][1], &full0[s], kb * kKB, 0);
        n0 = kb + 1;
      }
      // the ring lies over the first phase's stages: they are free once its MMAs have completed
      if (ok) ok = mbar_wait(&accf[0], 0, g.err);
      for (int p = 1; ok && p < nchain; ++p) {
        int K, N, wslot;
        phase_info(p, K, N, wslot);
        const int nkb = (K + kKB - 1) / kKB;
        for (int kb = 0; kb < nkb; ++kb, ++it) {
          const int s = it % NS;
          if (it >= NS && !mbar_wait(&emptyw[s], ((it / NS) - 1) & 1, g.err)) {
            ok = false;
            break;
          }
          unsigned char* st = ring + s * slotb;
          mbar_expect_tx(&fullw[s], 2u * (uint32_t)N * kKB * 2u);
          tma_load_2d(st, &mp.w[t][wslot][0], &fullw[s], kb * kKB, 0);
          tma_load_2d(st + halfb, &mp.w[t][wslot][1], &fullw[s], kb * kKB, 0);
        }
      }
      // the chunks' slots lie over everything the chain used
      if (ok) ok = mbar_wait(chain_done, 0, g.err);
      int nc_ = 0;
      for (int c = 0; ok && c < nch; ++c)
        for (int kb = 0; kb < nkc; ++kb) {
          const int s = nc_ % NC;
          if (nc_ >= NC && !mbar_wait(&emptyc[s], ((nc_ / NC) - 1) & 1, g.err)) {
            ok = false;
            break;
          }
          unsigned char* st = smem + chunk_slot(s);
          mbar_expect_tx(&fullc[s], 2 * kCHalf);  // rows beyond W_0 are zero-filled
          tma_load_2d(st, &mp.w[t][nh][0], &fullc[s], kb * kKB, CH * c);
          tma_load_2d(st + kCHalf, &mp.w[t][nh][1], &fullc[s], kb * kKB, CH * c);
          ++nc_;
        }
      // every copy this thread started has landed before the CTA may exit
      for (int kb = max(0, n0 - kP0); kb < n0; ++kb) mbar_wait(&full0[kb % kP0], (kb / kP0) & 1, g.err);
      for (int k = max(0, it - NS); k < it; ++k) mbar_wait(&fullw[k % NS], (k / NS) & 1, g.err);
      for (int k = max(0, nc_ - NC); k < nc_; ++k) mbar_wait(&fullc[k % NC], (k / NC) & 1, g.err);
    }
  } else if (warp == kMmaW) {
    {
      // ---- MMA issuer: the whole warp runs the loop, one lane issues ----
      const uint32_t by = elect_lane();
      bool ok = true;
      // three passes of one 16-column step: small terms first (lo.hi, hi.lo, then hi.hi)
      auto step = [&](uint32_t acc, uint64_t ah, uint64_t al, uint64_t bh, uint64_t bl, uint32_t idesc, bool first) {
        mma_f16_by(by, acc, al, bh, idesc, first ? 0 : 1);
        mma_f16_by(by, acc, ah, bl, idesc, 1);
        mma_f16_by(by, acc, ah, bh, idesc, 1);
      };
      {
        const uint32_t idesc = idesc_f16(SBM, g.width[1], 1);
        for (int kb = 0; kb < nk0; ++kb) {
          const int s = kb % kP0;
          if (!mbar_wait(&full0[s], (kb / kP0) & 1, g.err)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t sa = su32(smem + s * p0_stage);
          const uint64_t ah = sdesc_sw64(sa), al = sdesc_sw64(sa + kDHalf);
          const uint64_t bh = sdesc_sw64(sa + 2 * kDHalf), bl = sdesc_sw64(sa + 2 * kDHalf + halfb);
#pragma unroll
          for (int k = 0; k < kKB / 16; ++k)
            step(tmem, ah + 2 * k, al + 2 * k, bh + 2 * k, bl + 2 * k, idesc, (kb | k) == 0);
          mma_commit_by(by, &empty0[s]);
        }
        mma_commit_by(by, &accf[0]);
      }
      int it = 0;
      uint32_t free_par = 0, ready_par = 0;  // parities of the waits below, one bit per barrier
      if (nchain == 1) mma_commit_by(by, chain_done);
      for (int p = 1; ok && p < nchain; ++p) {
        int K, N, wslot;
        phase_info(p, K, N, wslot);
        const int buf = p & 1;
        // (the accumulator was last read two phases ago, by an epilogue that the operand blocks below have
        // waited for)
        const uint32_t idesc = idesc_f16(SBM, N, 1);
        const uint32_t acc = tmem + (uint32_t)(buf * 256);
        const int nkb = (K + kKB - 1) / kKB;
        for (int kb = 0; kb < nkb; ++kb, ++it) {
          const int s = it % NS;
          if ((kb & 1) == 0) {
            if (!mbar_wait(&aready[kb >> 1], (ready_par >> (kb >> 1)) & 1u, g.err)) {
              ok = false;
              break;
            }
            ready_par ^= 1u << (kb >> 1);
          }
          if (!mbar_wait(&fullw[s], (it / NS) & 1, g.err)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t sa = su32(smem + (kb >> 1) * kOpBlock), sw = su32(ring + s * slotb);
          const uint32_t ko = (uint32_t)(kb & 1) * 4;  // second half of the operand's 64-column block
          const uint64_t ah = sdesc_sw128(sa) + ko, al = sdesc_sw128(sa + 4 * kOpBlock) + ko;
          const uint64_t bh = sdesc_sw64(sw), bl = sdesc_sw64(sw + halfb);
#pragma unroll
          for (int k = 0; k < kKB / 16; ++k)
            step(acc, ah + 2 * k, al + 2 * k, bh + 2 * k, bl + 2 * k, idesc, (kb | k) == 0);
          mma_commit_by(by, &emptyw[s]);
        }
        mma_commit_by(by, &accf[buf]);
        if (p == nchain - 1) mma_commit_by(by, chain_done);
      }
      // chunks: the operand is complete (and the last chain accumulator, whose columns they take, is read)
      for (int kb = 0; ok && 2 * kb < nkc; ++kb) ok = mbar_wait(&aready[kb], (ready_par >> kb) & 1u, g.err);
      tc_fence_after();
      int nc_ = 0;
      for (int c = 0; ok && c < nch; ++c) {
        const int buf = c & 1;
        if (c >= 2) {
          if (!mbar_wait(&accfree[buf], (free_par >> buf) & 1u, g.err)) break;
          free_par ^= 1u << buf;
          tc_fence_after();
        }
        const uint32_t idesc = idesc_f16(SBM, min(CH, KD - CH * c), 1);
        const uint32_t acc = tmem + (uint32_t)(buf * CH);
        for (int kb = 0; kb < nkc; ++kb, ++nc_) {
          const int s = nc_ % NC;
          if (!mbar_wait(&fullc[s], (nc_ / NC) & 1, g.err)) {
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t sw = su32(smem + chunk_slot(s)), ah = tmem + 384u + (uint32_t)kb * 16u;
          const uint64_t al = sdesc_sw128(su32(smem + (4 + (kb >> 1)) * kOpBlock)) + (uint32_t)(kb & 1) * 4;
          const uint64_t bh = sdesc_sw64(sw), bl = sdesc_sw64(sw + kCHalf);
#pragma unroll
          for (int k = 0; k < kKB / 16; ++k) {
            mma_f16_by(by, acc, al + 2 * k, bh + 2 * k, idesc, (kb | k) != 0);
            mma_f16_ta_by(by, acc, ah + 8 * k, bl + 2 * k, idesc, 1);
            mma_f16_ta_by(by, acc, ah + 8 * k, bh + 2 * k, idesc, 1);
          }
          mma_commit_by(by, &emptyc[s]);
        }
        mma_commit_by(by, &accf[buf]);
      }
    }
  } else {
  // ---- epilogues: warps w and w + 4 own rows 32(w % 4) .. +31 and take 16-column pieces in turn ----
  const int quad = warp & 3, part = warp >> 2;
  const int rl = quad * 32 + lane;
  const long row = row0 + rl;
  const bool rv = row < row_end;
  const uint32_t tq = tmem + ((uint32_t)(quad * 32) << 16);
  int af[2] = {0, 0};  // accumulator-ready phases waited for, per buffer
  bool dead = false;   // after a timed-out wait: stop waiting, keep arriving
  auto wait_acc = [&](int buf) {
    if (!dead && !mbar_wait(&accf[buf], af[buf] & 1, g.err)) dead = true;
    ++af[buf];
    __syncwarp();
    tc_fence_after();
  };
  constexpr int kGroup = SBM * 8;  // floats of an 8-column group
  float* res = g.resid + (long)blockIdx.x * (SBM * kSLd) + rl * 8;
  auto gate_of = [&](int l) -> float* {
    return g.gate + ((long)l * gridDim.x + blockIdx.x) * (SBM * kSLd) + rl * 8;
  };
  // the next A operand: 64-column block kb of the high half at kb * kOpBlock, of the low half four blocks
  // further, row rl at rl * 128 bytes, 16-byte chunk j at (j ^ (rl % 8)) * 16 (128-byte swizzle); the chunks'
  // high half to tensor memory
  auto put_x = [&](int c, const float* x, bool chunks) {
    __align__(16) __nv_bfloat16 hi[16], lo[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) split2(x[i], hi[i], lo[i]);
    const int kb = c >> 6, j = (c & 63) >> 3;
    unsigned char* bh = smem + kb * kOpBlock + rl * 128;
    unsigned char* bl = bh + 4 * kOpBlock;
    if (chunks) {
      tmem_st8(tq + 384 + (c >> 1), reinterpret_cast<const uint32_t*>(hi));
      tmem_wait_st();
    } else {
      *reinterpret_cast<uint4*>(bh + ((j ^ (rl & 7)) << 4)) = *reinterpret_cast<const uint4*>(hi);
      *reinterpret_cast<uint4*>(bh + (((j + 1) ^ (rl & 7)) << 4)) = *reinterpret_cast<const uint4*>(hi + 8);
    }
    *reinterpret_cast<uint4*>(bl + ((j ^ (rl & 7)) << 4)) = *reinterpret_cast<const uint4*>(lo);
    *reinterpret_cast<uint4*>(bl + (((j + 1) ^ (rl & 7)) << 4)) = *reinterpret_cast<const uint4*>(lo + 8);
  };
  // after this thread's second piece of a 64-column block: its part of the block is written and its
  // accumulator columns are in registers
  auto block_done = [&](int k) {
    if (!(k & 1)) return;
    fence_async_smem();
    tc_fence_before();
    mbar_arrive(&aready[k >> 1]);
  };
  auto load16 = [&](const float* base, int c, float* y) {
    ld_v8(base + (c >> 3) * kGroup, y);
    ld_v8(base + ((c >> 3) + 1) * kGroup, y + 8);
  };
  auto store16 = [&](float* base, int c, const float* y) {
    st_v8(base + (c >> 3) * kGroup, y);
    st_v8(base + ((c >> 3) + 1) * kGroup, y + 8);
  };
  // biases and output weights of this tile's type into shared memory
  for (int l = 0; l < nh; ++l)
    for (int c = threadIdx.x; c < 256; c += kSEpi)
      s_bias[l * 256 + c] = c < g.width[l + 1] ? __ldg(g.bias[t][l] + c) : 0.f;
  for (int c = threadIdx.x; c < 256; c += kSEpi) s_wl[c] = c < g.width[nh] ? __ldg(g.w_last[t] + c) : 0.f;
  bar_sync(1, kSEpi);
  // forward
  for (int l = 0; l < nh; ++l) {
    const int N = g.width[l + 1], nc = (N + 63) & ~63;  // zeros to the next whole block: the operand's K padding
    const bool last = (l == nh - 1), sk = g.skip[l] == 1;
    const float* bias = s_bias + l * 256;
    float e_acc = 0.f;
    // the accumulator (and residual) pieces load one ahead of the piece being processed
    uint32_t na[16];
    float ny[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) ny[i] = 0.f;
    if (sk) load16(res, part * 16, ny);
    wait_acc(l & 1);
    const uint32_t ta = tq + (uint32_t)((l & 1) * 256);
    tmem_ld16_async(ta + part * 16, na);
    tmem_wait_ld();
    for (int c = part * 16, k = 0; c < nc; c += kStep, ++k) {
      uint32_t ra[16];
      float ry[16];
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        ra[i] = na[i];
        ry[i] = ny[i];
      }
      if (c + kStep < nc) {
        tmem_ld16_async(ta + c + kStep, na);
        if (sk && c + kStep < N) load16(res, c + kStep, ny);
      }
      float out[16], y[16], gt[16];
      if (c < N) {  // widths are multiples of 16: a piece is all real columns or all padding
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          const int col = c + i;
          const float th = tanh_ex(__uint_as_float(ra[i]) + bias[col]);
          y[i] = th + (sk ? ry[i] : 0.f);
          gt[i] = 1.f - th * th;
          if (last) {
            const float w = s_wl[col];
            e_acc += y[i] * w;
            out[i] = w * gt[i];
          } else {
            out[i] = y[i];
          }
        }
      } else {
#pragma unroll
        for (int i = 0; i < 16; ++i) out[i] = 0.f;
      }
      tmem_wait_ld();  // the next piece has landed
      put_x(c, out, nh == 1);
      block_done(k);
      if (!last && c < N) {
        store16(res, c, y);  // the residual stream of the next layer
        store16(gate_of(l), c, gt);
      }
    }
    if (last) {
      s_e[part * SBM + rl] = e_acc;
      bar_sync(1, kSEpi);
      if (part == 0 && rv) {
        float e = 0.f;
#pragma unroll
        for (int q = 0; q < kParts; ++q) e += s_e[q * SBM + rl];
        g.atom_e[g.perm[row]] = (double)(e + g.b_last[t]);
      }
    }
  }
  // backward of layers nh-1 .. 1: gz_{l-1} as the next operand, gy_{l-1} kept for the next skip
  for (int l = nh - 1; l >= 1; --l) {
    const int N = g.width[l], nc = (N + 63) & ~63;
    const bool top = (l == nh - 1), sk = g.skip[l] == 1, keep = (l - 1 >= 1);
    const int p = nh + (nh - 1 - l);  // phase index
    const bool ldy = sk && !top;
    const float* gates = gate_of(l - 1);
    uint32_t na[16];
    float ny[16], ng[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) ny[i] = 0.f;
    if (ldy) load16(res, part * 16, ny);
    load16(gates, part * 16, ng);
    wait_acc(p & 1);
    const uint32_t ta = tq + (uint32_t)((p & 1) * 256);
    tmem_ld16_async(ta + part * 16, na);
    tmem_wait_ld();
    for (int c = part * 16, k = 0; c < nc; c += kStep, ++k) {
      uint32_t ra[16];
      float ry[16], gt[16];
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        ra[i] = na[i];
        ry[i] = ny[i];
        gt[i] = c < N ? ng[i] : 0.f;
      }
      if (c + kStep < nc) {
        tmem_ld16_async(ta + c + kStep, na);
        if (c + kStep < N) {
          if (ldy) load16(res, c + kStep, ny);
          load16(gates, c + kStep, ng);
        }
      }
      float gy[16], gz[16];
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        const int col = c + i;
        float v = col < N ? __uint_as_float(ra[i]) : 0.f;
        if (sk && col < N) v += top ? s_wl[col] : ry[i];
        gy[i] = v;
        gz[i] = v * gt[i];
      }
      tmem_wait_ld();
      put_x(c, gz, l == 1);
      block_done(k);
      if (keep && c < N) store16(res, c, gy);
    }
  }
  // dE/dD in chunks of 192 columns from the two alternating accumulators: stored, or (gT mode, 16-column
  // pieces = one m) folded at once into dE/dT, term 1 per piece and term 2 accumulated per row
  const bool gtm = g.gT != nullptr;
  float ext[16][4];
#pragma unroll
  for (int l = 0; l < 16; ++l)
#pragma unroll
    for (int q = 0; q < 4; ++q) ext[l][q] = 0.f;
  float4 tl[16];  // T_< of this thread's row
#pragma unroll
  for (int l = 0; l < 16; ++l)
    tl[l] = gtm && rv ? __ldg(reinterpret_cast<const float4*>(g.Tm + (row * g.M + l) * 4))
                      : make_float4(0.f, 0.f, 0.f, 0.f);
  for (int c = 0; c < nch; ++c) {
    const int buf = c & 1;
    wait_acc(buf);
    const int N = min(CH, KD - CH * c);
    const uint32_t tb = tq + (uint32_t)(buf * CH);
    for (int q = part * 16; q < N; q += kStep) {
      float v[16];
      tmem_ld16(tb + q, v);
      if (rv) {
        if (gtm) {
          const int m = (CH * c + q) >> 4;
          const float4 tm = __ldg(reinterpret_cast<const float4*>(g.Tm + (row * g.M + m) * 4));
          float t1[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
          for (int l = 0; l < 16; ++l) {
            t1[0] += v[l] * tl[l].x;
            t1[1] += v[l] * tl[l].y;
            t1[2] += v[l] * tl[l].z;
            t1[3] += v[l] * tl[l].w;
            ext[l][0] += v[l] * tm.x;
            ext[l][1] += v[l] * tm.y;
            ext[l][2] += v[l] * tm.z;
            ext[l][3] += v[l] * tm.w;
          }
          reinterpret_cast<float4*>(g.gT)[(long)m * rows + row] = make_float4(t1[0], t1[1], t1[2], t1[3]);
        } else {
          float* dst = g.gD + row * KD + CH * c + q;
          st_v8(dst, v);
          st_v8(dst + 8, v + 8);
        }
      }
    }
    tc_fence_before();
    mbar_arrive(&accfree[buf]);
  }
  if (gtm) {
    // term 2 of the rows' first 16 m: the parts' partial sums meet in the operand buffer (every MMA of
    // the tile completed before the last chunk's accumulator became ready).  A row's dE/dT of m < 16 was
    // written by the thread of m's parity, which is the one that adds here.
    float* s_ext = reinterpret_cast<float*>(smem);  // [kParts][128][68]
#pragma unroll
    for (int l = 0; l < 16; ++l)
      *reinterpret_cast<float4*>(s_ext + ((part * SBM) + rl) * 68 + l * 4) =
          make_float4(ext[l][0], ext[l][1], ext[l][2], ext[l][3]);
    bar_sync(1, kSEpi);
    if (rv) {
      float4 a[16 / kParts];
#pragma unroll
      for (int i = 0; i < 16 / kParts; ++i)
        a[i] = reinterpret_cast<float4*>(g.gT)[(long)(part + kParts * i) * rows + row];
#pragma unroll
      for (int i = 0; i < 16 / kParts; ++i) {
        const int l = part + kParts * i;
#pragma unroll
        for (int pp = 0; pp < kParts; ++pp) {
          const float4 e = *reinterpret_cast<const float4*>(s_ext + ((pp * SBM) + rl) * 68 + l * 4);
          a[i].x += e.x;
          a[i].y += e.y;
          a[i].z += e.z;
          a[i].w += e.w;
        }
        reinterpret_cast<float4*>(g.gT)[(long)l * rows + row] = a[i];
      }
    }
  }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == kProd) tmem_dealloc(tmem, 512);
}

// the buffer, barriers, energies, biases and output weights
size_t split_smem(int rows) {
  return (size_t)buffer_bytes(rows) + (2 * kP0 + 6 + 2 + 2 + 4 + 1 + 2 * kCRing + 1) * 8 + 16 + (kParts * SBM + kSL * 256 + 256) * 4 + 1024;
}

}  // namespace

bool fit_split_supported(const DeviceModel& m) {
  const int nfl = m.n_fit_layers, nh = nfl - 1;
  if (nh < 1 || nh > kSL) return false;
  const int KD = m.M * m.A;
  if (KD % 16 != 0) return false;
  for (int t = 0; t < m.cfg.ntypes; ++t)
    for (int l = 0; l < nh; ++l) {
      const LayerDesc& L = m.fit[(size_t)t * nfl + l];
      const LayerDesc& L0 = m.fit[l];
      if (L.n_in != L0.n_in || L.n_out != L0.n_out || L.skip != L0.skip) return false;
      if (L.n_out % 16 || L.n_out > 256 || L.skip > 1 || (l == 0 && L.skip)) return false;
    }
  return m.fit[0].n_in == KD && m.fit_wt_bf16_lo != nullptr;
}

int run_fitting_split(const DeviceModel& m, const PathConst& pc, const __nv_bfloat16* Dhi, const __nv_bfloat16* Dlo,
                      const PathIO& io, Arena& ar, cudaStream_t st, const float** gD_out, const float* Tm,
                      float* gT) {
  const long N = pc.natoms;
  const int nfl = m.n_fit_layers, nh = nfl - 1;
  const int nt = pc.ntypes;
  const int KD = pc.M * pc.A;
  const bool gtm = gT != nullptr && Tm != nullptr && pc.A == 16;
  const long max_tiles = (N + SBM - 1) / SBM + nt;  // every type's last tile may be short
  float* resid = ar.get<float>(max_tiles * SBM * kSLd);
  float* gate = ar.get<float>((long)nh * max_tiles * SBM * kSLd);
  float* gD = gtm ? nullptr : ar.get<float>(N * KD);
  if (ar.measure) return DP_OK;
  if (!ar.ok()) {
    set_error("scratch allocation failed");
    return DP_E_OOM;
  }
  SplitArgs a;
  std::memset(&a, 0, sizeof(a));
  a.ntypes = nt;
  a.nh = nh;
  a.width[0] = KD;
  for (int l = 0; l < nh; ++l) {
    a.width[l + 1] = m.fit[l].n_out;
    a.skip[l] = m.fit[l].skip;
  }
  int maxw = 0;
  for (int l = 0; l < nh; ++l) maxw = std::max(maxw, a.width[l + 1]);
  a.rows = slot_rows(maxw);
  int tiles = 0;
  for (int t = 0; t <= nt; ++t) {
    a.row_start[t] = io.type_start[t];
    a.tile_start[t] = tiles;
    if (t < nt) tiles += (io.type_start[t + 1] - io.type_start[t] + SBM - 1) / SBM;
  }
  SplitMaps mp;
  std::memset(&mp, 0, sizeof(mp));
  int rc = make_tmap_bf16(&mp.d[0], Dhi, N, KD, SBM, kKB);
  if (rc == DP_OK) rc = make_tmap_bf16(&mp.d[1], Dlo, N, KD, SBM, kKB);
  if (rc != DP_OK) return rc;
  const float* p32 = m.p32;
  for (int t = 0; t < nt; ++t) {
    for (int l = 0; l < nh; ++l) {
      const LayerDesc& L = m.fit[(size_t)t * nfl + l];
      a.bias[t][l] = p32 + L.w_off + (long)L.n_in * L.n_out;
      for (int hl = 0; hl < 2; ++hl) {
        const CUtensorMap* f = fit_weight_map(m, t, l, 0, L.n_out, hl == 1, kKB);
        const CUtensorMap* b = l == 0 ? fit_weight_map(m, t, 0, 1, CH, hl == 1, kKB) : fit_weight_map(m, t, l, 1, L.n_in, hl == 1, kKB);
        if (!f || !b) return DP_E_CUDA;
        mp.w[t][l][hl] = *f;
        mp.w[t][nh + l][hl] = *b;
      }
    }
    const LayerDesc& Lo = m.fit[(size_t)t * nfl + nh];
    a.w_last[t] = p32 + Lo.w_off;
    a.b_last[t] = m.fit_out_bias[t];
  }
  a.resid = resid;
  a.gate = gate;
  a.perm = io.perm;
  a.atom_e = io.atom_energy;
  a.gD = gD;
  a.gT = gtm ? gT : nullptr;
  a.Tm = Tm;
  a.M = pc.M;
  a.err = &io.status->timeout;
  if (tiles > 0) {
    ProfScope _ps(io.prof, "fit_split_tc", st);
    const size_t smem = split_smem(a.rows);
    DP_CUDA_TRY(allow_max_smem(k_fit_split));
    k_fit_split<<<tiles, kSThreads, smem, st>>>(mp, a);
    DP_CUDA_TRY(cudaGetLastError());
  }
  *gD_out = gD;
  return DP_OK;
}

}  // namespace dpgb
