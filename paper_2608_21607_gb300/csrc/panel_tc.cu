// Fused Z-panel contraction and dense loss pass on the tcgen05 tensor cores.
//
// For M-side rows m_i (a tile of 128) and Q-side rows q_k (streamed in
// chunks of BN), the panel kernel computes, without writing any tile of L or
// Z to global memory (the fused kernel of Sec. 4.2, eq. "kernel"):
//   L_ik = m_i . q_k                         MMA1: TMEM <- W tile x chunk^T
//   P_ik = min(0, L_ik)      (Z form, eq. updateZ)   -- epilogue in registers,
//        = -max(0, L_ik)     (Delta form, eq. updateD)  written back to TMEM
//   R_i  = sum_k P_ik q_k                    MMA2: TMEM R += P (TMEM) x chunk
// The same shared-memory copy of each chunk feeds both products: K-major for
// MMA1 and MN-major for MMA2.  The W tile is MMA1's A operand from shared
// memory (bf16 mode, TMA-loaded with the chunk's swizzle) or from TMEM
// (fp32-accurate mode, written by the epilogue warps).  Every factor has bf16
// pieces hi = bf16(x), lo = bf16(x - hi), lo2 = bf16(x - hi - lo).  bf16 mode:
// both products use hi alone (the Gram matrix and the support term are formed
// from the same rounded rows, so that the rounding of q is not a coherent error
// that the solve would amplify).  fp32-accurate mode (SPLIT): MMA1 = w_hi q_hi +
// w_hi q_lo + w_lo q_hi, P = P_hi + P_lo, MMA2 = P_hi (q_hi + q_lo + q_lo2) +
// P_lo q_hi.
//
// The loss kernel runs MMA1 only, over all of W against all of B, and sums
// max(0, L)^2 and max(0, L) over the entries outside the support of S (the
// dense parts of eq. SLloss / eq. RMSE / eq. WJD); the support entries are
// summed by a separate pass.  139,255 rows on both sides at r = 64: 5.6 ms of
// dense pass against 1.3 ms of tensor work; the rest is the epilogue's sums
// and, on rows of many entries, finding the support columns (3.5 ms with one
// entry a row).
//
// Warp roles (352 threads, one CTA per SM, persistent over M tiles):
//   warps 0-7  epilogue, two warpgroups; in each, thread t owns TMEM lane t =
//              tile row t
//   warp 8     TMA producer of Q chunks and W tiles (+ TMEM allocation)
//   warp 9     issues MMA1 (L = W Q^T) for every chunk
//   warp 10    issues MMA2 (R += P Q) for every chunk
// The MMA warps run converged and predicate each tcgen05 operation on an
// elected lane.
// With two of them the bookkeeping of one (barrier tests, votes, branches: about
// 200 cycles per chunk) runs while the other's MMAs keep the tensor core busy,
// whose queue holds next to nothing.  (One warp for both was faster, 93 against
// 100 us at r_pad = 64 and 158 against 183 us at r_pad = 128, 139,255 rows
// against 4,096, only without the wait on b_lfree, that is, by relying on an
// order between products into different accumulators that PTX does not give.)
// Every mbarrier wait is bounded (2 s): on expiry the kernel records
// NMD_ERR_TIMEOUT, the other roles stop at their next wait, in-flight MMAs
// and copies are drained and TMEM is freed before the kernel returns.
#include <cudaTypedefs.h>
#include <limits.h>

#include <algorithm>
#include <map>
#include <mutex>
#include <tuple>

#include "nmd_internal.cuh"
#include "tc_ptx.cuh"

namespace nmd {
namespace {

using namespace tc;

constexpr int kEpiThreads = 256;                 // two epilogue warpgroups
constexpr int kProducerWarp = 8, kMma1Warp = 9, kMma2Warp = 10;
constexpr int kThreads = 352;
// The panel kernel's registers are capped, so that an update block fits beside
// it on an SM: three of its warps on a sub-partition and two of the update's
// (of 72 registers in the bf16 mode at r_pad = 64) within 16,384 registers.
// 120 where that is as far as it goes (bf16, r_pad = 64: 139,255 rows, blocks of
// 4,096, 9.04 ms a sweep, 9.10 at 112, 9.57 at 104, which spills, 10.93 at 128,
// where the deferred update no longer runs beside it).
// The fp32-accurate kernel of r_pad = 64 has 128, without which it spills: 23.5 ms
// a sweep of the same shape, 24.15 at 112.
constexpr int BM = 128;
constexpr uint64_t kTimeoutNs = 2000000000ull;

// SK: a chunk-skipping kernel (its chunk size is part of what
// nmd_range_mask and nmd_skip_count report)
template <int RP, bool SPLIT, bool LOSS, bool SK = false>
struct Cfg {
  // fp32-accurate mode at r_pad = 256: W hi + lo take 256 TMEM columns, so a
  // CTA accumulates one 128-column half of R (blockIdx.y selects it) and the
  // first product is formed once per half
  static constexpr bool RHALF = SPLIT && !LOSS && RP == 256;
  static constexpr int NR = RHALF ? RP / 2 : RP;        // R columns of one CTA
  // TMEM columns of one R accumulator; the loss pass has none.  In the bf16
  // mode the second product multiplies P by q_hi alone: the update pairs
  // this term with the Gram matrix of q_hi, so the rounding of q cancels
  // (see update_kernel), and R needs one accumulator of r_pad columns.
  static constexpr int RCOLS = LOSS ? 0 : NR;
  // bf16 mode, r_pad <= 128: the W tile is the first product's A operand
  // from shared memory (loaded by TMA) instead of TMEM, which leaves TMEM
  // to the L buffers.
  static constexpr bool WSMEM = !SPLIT && !LOSS && RP <= 128;
  // Q rows per chunk (the N of the first product and the K of the second):
  // 128 where at least two L buffers of 128 columns fit beside R and W, else
  // 64.  A chunk of 64 rows reads the W tile from shared memory twice as
  // often per product, which at r_pad = 128 takes longer than the product.
  static constexpr int BN = WSMEM ? (RP == 128 && SK ? 64 : 128)
                                  : ((RP == 256 || (SPLIT && RP == 128)) ? 64 : 128);
  // TMEM columns of one W tile (hi [+ lo]); none when it sits in shared memory
  static constexpr int WCOLS = WSMEM ? 0 : (SPLIT ? RP : RP / 2);
  static constexpr int W_BYTES = WSMEM ? BM * RP * 2 : 0;   // one W tile in shared memory
  static constexpr int NWB = (RP == 256) ? 1 : 2;      // W tile buffers
  static constexpr int FREE = 512 - NWB * WCOLS - RCOLS;
  static constexpr int NB_MAX = LOSS ? 6 : (RP == 128 && !SPLIT && !SK ? 2 : 3);
  static constexpr int NB = FREE / BN >= NB_MAX ? NB_MAX : FREE / BN;  // L buffers
  // R accumulators: with two, the second product of the next tile starts
  // while the epilogue still reads this tile's R
  static constexpr int NRB = (!LOSS && NB * BN + 2 * RCOLS + NWB * WCOLS <= 512) ? 2 : 1;
  // with two L buffers both epilogue warpgroups share every chunk (half of
  // its columns each), which halves the time a buffer is held; with three
  // they take alternate chunks (fewer hand-offs per element)
  static constexpr bool HALF = !LOSS && NB == 2;
  static constexpr int PANEL_W = RP < 64 ? RP : 64;    // elements per row of one swizzle panel
  static constexpr int ROWB = PANEL_W * 2;             // bytes per panel row (= swizzle width)
  static constexpr int PANEL_BYTES = BN * ROWB;
  static constexpr int NPANEL = RP / PANEL_W;
  static constexpr int OPER_BYTES = BN * RP * 2;       // one bf16 piece of a chunk
  // bf16 pieces of each chunk in shared memory: hi in the bf16 mode, hi, lo
  // and lo2 in the fp32-accurate mode (hi and lo in its loss pass)
  static constexpr int NQ = SPLIT ? (LOSS ? 2 : 3) : 1;
  static constexpr int STAGE_BYTES = OPER_BYTES * NQ;
  // R on its way out: 32 rows x 32 columns per epilogue warp
  static constexpr int STG_BYTES = LOSS ? 0 : (kEpiThreads / 32) * 4096;
  // stages within 160 KB with the W tiles and the R staging (r_pad <= 64: 165
  // KB in all, so that an update block fits beside the CTA), 224 KB at r_pad =
  // 128; beside the staging where W sits in TMEM
  static constexpr int NSTAGE_RAW =
      (WSMEM ? (RP <= 64 ? 160 : 224) * 1024 - NWB * W_BYTES - STG_BYTES : 160 * 1024) / STAGE_BYTES;
  static constexpr int NSTAGE = NSTAGE_RAW > 8 ? 8 : (NSTAGE_RAW < 2 ? 2 : NSTAGE_RAW);
  static constexpr uint32_t SWZ = PANEL_W == 64 ? SWZ_128B : (PANEL_W == 32 ? SWZ_64B : SWZ_32B);
  // shared memory: stages, W tiles (WSMEM), R staging, barriers, TMEM slot + abort flag, ...
  static constexpr size_t OFF_W = (size_t)NSTAGE * STAGE_BYTES;
  static constexpr int W_PANEL_BYTES = BM * ROWB;     // one swizzle panel of a W tile
  static constexpr size_t OFF_STG = OFF_W + (size_t)NWB * W_BYTES;
  // loss pass: each epilogue thread's window of column indices (32, at a stride of 33)
  static constexpr size_t OFF_WIN = OFF_STG;
  static constexpr int WIN_BYTES = LOSS ? kEpiThreads * 33 * 4 : 0;
  static constexpr size_t OFF_BARS = OFF_STG + STG_BYTES + WIN_BYTES;
  static constexpr int COL_L = 0;                     // NB x BN columns
  static constexpr int COL_R = NB * BN;               // NRB x RCOLS columns
  static constexpr int COL_W = COL_R + NRB * RCOLS;   // NWB x WCOLS columns
  // barriers: full[NSTAGE], empty[NSTAGE], lfull[NB], pfull[NB], lfree[NB], rfull[2], rempty[2],
  // wfull[2], wempty[2], drain, drain2
  static constexpr int NBAR = 2 * NSTAGE + 3 * NB + 10;
  // after the barriers: TMEM slot and abort flag (64 B), the loss reduction
  // (256 x 16 B), and 8 flags per L buffer (Delta form: P nonzero per warp)
  static constexpr size_t SMEM_USED = 1024 + OFF_BARS + NBAR * 8 + 64 + (LOSS ? 256 * 16 : 0) + NB * 32;
  // at least 120 KB so that a second CTA (and its 512-column TMEM request)
  // never shares the SM
  static constexpr size_t SMEM = SMEM_USED > 120 * 1024 ? SMEM_USED : 120 * 1024;
  static_assert(NB >= 2, "need two L buffers");
  static_assert(NSTAGE >= 2, "stages");
  static_assert(SMEM <= 227 * 1024, "shared memory per block");
  static_assert(COL_W + NWB * WCOLS <= 512, "TMEM budget");
  static_assert(LOSS || COL_R + (NRB - 1) * RCOLS + (RCOLS + 31) / 32 * 32 <= 512, "R is read 32 columns at a time");
  static_assert(BN % 32 == 0 && RP % 16 == 0, "shapes");
};

struct TcParams {
  int64_t m0, M;        // M-side rows [m0, m0 + M) of the M factor
  int64_t q0, K;        // Q-side rows [q0, q0 + K) of the Q factor
  const bf16* Mhi;      // M factor operand copies (absolute row index)
  const bf16* Mlo;
  float* R;             // M x RP output (panel kernel)
  double* parts;        // per-CTA loss partials (loss kernel)
  int* status;
  float* Lout;          // verification: raw L (M x K, row-major) or nullptr
  const int64_t* rowptr;   // loss kernel: CSR of S, whose entries the dense pass skips
  const int32_t* cidx;
  unsigned long long* skips;   // Delta form: count of chunks whose second product was skipped (or nullptr)
  int skip_on;                 // Delta form: skip chunks whose rectified tile is zero
  // split K (steps with fewer tiles than SMs): CTA z takes Q-side rows
  // [q0 + z ksplit, ...) and writes its partial R at R + z rstride
  int64_t ksplit;              // 0: no split
  int64_t rstride;
  // range-search skipping (Delta form): bit c of tile t's words
  // rmask[t rwords ...] set = Q chunk c of the step is all L <= 0 for the
  // tile's rows (see range_mask_kernel); nullptr: no chunk is skipped
  const uint32_t* rmask;
  int64_t rwords;
  // nearest-neighbour pass (M side = Q side = one point set): per row the
  // largest L_ij over j != i, as an orderable key (value bits << 32 |
  // ~j); the caller zeroes the keys
  unsigned long long* nn_key;
  // update pass (M side = the step's right-hand side R, Q side = G^{-1}):
  // X = (R + Rs) G^{-1} with R and Rs fp32 rows (relative to the range, Rs
  // only where upd_flags is set) split into two bf16 pieces as they are
  // loaded; the epilogue applies the update of eqs. lsqA_sto / spLsqA to the
  // factor rows upd_row0 + i of upd_M (fp32 master), upd_E (momentum) and
  // upd_hi (bf16 piece)
  const float* upd_R;
  const float* upd_Rs;
  const uint8_t* upd_flags;
  float* upd_M;
  float* upd_E;
  bf16* upd_hi;
  int64_t upd_row0;
  float eta, gamma;
  int momentum, delta_form;
};

__device__ __forceinline__ void record(int* status, int code, int detail) {
  if (atomicCAS(status, 0, code) == 0) status[1] = detail;
}

// Bounded wait on an mbarrier phase.  Returns false if the kernel is aborting.
// The polls suspend in hardware until the phase completes (or 20 us pass), so
// waiting warps do not take issue slots from the MMA and copy threads.
__device__ __noinline__ bool wait_bar_slow(uint32_t bar, uint32_t parity, volatile int* abort_flag, int* status,
                                           int where, uint64_t limit_ns = kTimeoutNs) {
  const uint64_t t0 = globaltimer_ns();
  for (;;) {
    if (mbar_try_wait(bar, parity)) return true;
    if (*abort_flag) return false;
    if (globaltimer_ns() - t0 > limit_ns) {
      *abort_flag = 1;
      record(status, NMD_ERR_TIMEOUT, where);
      return false;
    }
  }
}
__device__ __forceinline__ bool wait_bar(uint32_t bar, uint32_t parity, volatile int* abort_flag, int* status,
                                         int where) {
  if (mbar_try_wait(bar, parity)) return true;
  return wait_bar_slow(bar, parity, abort_flag, status, where);
}

// Wait of a converged warp, every lane testing the phase: `ready` is the
// result of an earlier mbar_test_wait (a test takes about 60 cycles even when
// the phase is complete, so the MMA warp starts it ahead of the instructions
// it does not guard).
__device__ __forceinline__ bool conv_wait(bool ready, uint32_t bar, uint32_t parity, volatile int* abort_flag,
                                          int* status, int where) {
  if (__all_sync(0xffffffffu, ready)) return true;
  const bool ok = wait_bar_slow(bar, parity, abort_flag, status, where);
  return __all_sync(0xffffffffu, ok);
}
__device__ __forceinline__ bool conv_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag, int* status,
                                          int where) {
  return conv_wait(mbar_try_wait(bar, parity), bar, parity, abort_flag, status, where);
}

// The live Q chunks [0, n) of one tile (this CTA's split of it starts at
// chunk c0 of the tile's mask): those whose mask bit is clear.  A tile whose
// chunks are all masked still computes its chunk 0, which gives R = 0 (its L
// is <= 0 throughout), so that every tile has a first and a last chunk and
// the R hand-off is the same as without skipping.  The first 64 chunks'
// bits are kept in a register (a stochastic step has at most 64 chunks).
struct ChunkMask {
  const uint32_t* m;   // the tile's words, or nullptr (every chunk live)
  int64_t c0;
  bool none;           // every chunk masked
  uint64_t live64;     // bit c: chunk c (< 64) is live
  __device__ __forceinline__ bool masked_far(int64_t c) const {
    const int64_t b = c0 + c;
    return (m[b >> 5] >> (b & 31)) & 1u;
  }
  __device__ __forceinline__ bool live(int64_t c) const {
    if (m == nullptr) return true;
    if (none) return c == 0;
    return c < 64 ? ((live64 >> c) & 1ull) != 0 : !masked_far(c);
  }
};

template <bool RANGE>
__device__ __forceinline__ ChunkMask chunk_mask(const TcParams& p, int64_t t, int64_t c0, int64_t n,
                                                int64_t* last, int64_t* nlive) {
  ChunkMask cm{nullptr, c0, false, ~0ull};
  *last = n - 1;
  *nlive = n;
  if (!RANGE || p.rmask == nullptr) return cm;
  cm.m = p.rmask + t * p.rwords;
  // bits c0 .. c0 + 63 of the tile's words (words past the end read as masked)
  const int64_t w = c0 >> 5;
  const int sh = (int)(c0 & 31);
  const uint32_t w0 = w < p.rwords ? cm.m[w] : ~0u;
  const uint32_t w1 = w + 1 < p.rwords ? cm.m[w + 1] : ~0u;
  const uint32_t w2 = w + 2 < p.rwords ? cm.m[w + 2] : ~0u;
  const uint64_t lo = ((uint64_t)w1 << 32) | w0;
  const uint64_t bits = sh ? (lo >> sh) | ((uint64_t)w2 << (64 - sh)) : lo;
  const uint64_t inrange = n >= 64 ? ~0ull : ((1ull << n) - 1ull);
  cm.live64 = ~bits & inrange;
  int64_t cnt = __popcll(cm.live64), lst = cm.live64 ? 63 - __clzll(cm.live64) : -1;
  for (int64_t c = 64; c < n; ++c)
    if (!cm.masked_far(c)) {
      ++cnt;
      lst = c;
    }
  cm.none = cnt == 0;
  *last = cm.none ? 0 : lst;
  *nlive = cm.none ? 1 : cnt;
  return cm;
}

// The live chunks of a CTA's tiles in order, as an MMA warp walks them: whether
// the current chunk is its tile's first or last live one.  Without a
// range-search mask this is a counter within the tile.
template <bool RANGE>
struct ChunkWalk {
  int left, n, c, clast;   // tiles left (this one included), chunks per tile, current and last live chunk
  bool first;
  int t;                   // RANGE: the tile, its mask
  int64_t kc0, nlive;
  ChunkMask cm;
  __device__ __forceinline__ ChunkWalk(const TcParams& p, int ntiles, int nchunks, int64_t kc0_)
      : left((ntiles - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x), n(nchunks), t(blockIdx.x), kc0(kc0_) {
    enter(p);
  }
  __device__ __forceinline__ void enter(const TcParams& p) {
    c = 0;
    first = true;
    clast = n - 1;
    if (!RANGE || left <= 0) return;
    int64_t last;
    cm = chunk_mask<RANGE>(p, t, kc0, n, &last, &nlive);
    clast = (int)last;
    while (!cm.live(c)) ++c;
  }
  __device__ __forceinline__ bool valid() const { return left > 0; }
  __device__ __forceinline__ bool last() const { return c == clast; }
  __device__ __forceinline__ void next(const TcParams& p) {
    if (!RANGE) {   // (no branches: n >= 1)
      first = c == clast;
      left -= first ? 1 : 0;
      c = first ? 0 : c + 1;
      return;
    }
    if (last()) {
      --left;
      t += gridDim.x;
      enter(p);
      return;
    }
    first = false;
    ++c;
    while (!cm.live(c)) ++c;
  }
};

// R of one 128-row tile from TMEM to global memory by one epilogue warp (rows
// [li0, li0 + 32) of the step, lanes [lane_base ...) of TMEM): 32 columns at a
// time through the warp's 4 KB of shared memory (16-byte pieces swizzled by
// row), so that a store instruction covers whole 128-byte lines of four rows.
// (Written straight from the TMEM layout, one row per lane, every 16-byte
// store of a warp touched 32 lines: about 3,500 cycles per tile at r_pad = 64,
// a tenth of the tile's time.)  Warpgroup wg takes every second group of 32
// columns; the warp's last TMEM read releases the accumulator (b_rempty)
// before the stores.  Called once per tile and warp, and kept out of line: the
// hot loops of the epilogue and MMA warps then stay in the instruction caches.
template <int NR, int RP>
__device__ __noinline__ void store_r_tile(uint32_t tmem_r, uint32_t b_rempty, float* stg, float* dst, int64_t li0,
                                          int64_t M, int wg, int lane) {
  constexpr int NJ = (NR + 31) / 32;
#pragma unroll 1
  for (int j = wg; j < NJ; j += 2) {
    uint32_t v[32];
    tmem_ld32(tmem_r + j * 32, v);   // RP = 16 reads 16 columns past R
    tmem_wait_ld(v);
    if (j + 2 >= NJ) {
      fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(b_rempty);
    }
#pragma unroll
    for (int k = 0; k < 8; ++k)
      *(uint4*)(stg + lane * 32 + ((k ^ (lane & 7)) << 2)) = make_uint4(v[4 * k], v[4 * k + 1], v[4 * k + 2], v[4 * k + 3]);
    __syncwarp();
    const int ch = lane & 7;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int rr = 4 * u + (lane >> 3);
      if (li0 + rr < M && j * 32 + 4 * ch < NR)
        *(float4*)(dst + (int64_t)rr * RP + j * 32 + 4 * ch) = *(const float4*)(stg + rr * 32 + ((ch ^ (rr & 7)) << 2));
    }
    __syncwarp();   // the buffer is refilled by the next 32 columns
  }
  if (wg >= NJ) {   // no columns for this warpgroup (r_pad <= 32): release at once
    fence_before();
    __syncwarp();
    if (lane == 0) mbar_arrive(b_rempty);
  }
}

// MODE: 0 the panel contraction R = P(L) Q; 1 the loss pass (first product
// only, sums of max(0, L)^2 and max(0, L) off the support); 2 the nearest-
// neighbour pass (first product only, per row the largest L_ij, j != i);
// 3 the update pass (first product only: X = R G^{-1} and the step applied
// to the factor rows in the epilogue).
// SKIPM (Delta form only): 1 skips the second product of chunks whose
// rectified tile is zero (a vote of the epilogue warps); 2 skips both
// products of the chunks that the range-search mask clears.  Separate
// instantiations, so that the kernel without them carries none of the checks.
template <int RP, int EPI, bool SPLIT, int MODE, int SKIPM>
__global__ void __maxnreg__(MODE == 0 ? (RP <= 32 || (RP == 64 && SPLIT) ? 128 : RP == 64 ? 120 : 112) : 168)
    panel_tc_kernel(const __grid_constant__ CUtensorMap tq_hi, const __grid_constant__ CUtensorMap tq_lo,
                    const __grid_constant__ CUtensorMap tq_lo2, const __grid_constant__ CUtensorMap tw,
                    const TcParams p) {
  constexpr bool LOSS = MODE != 0;     // the first product only
  constexpr bool SUMS = MODE == 1, NEAREST = MODE == 2, UPDATE = MODE == 3;
  static_assert(!UPDATE || SPLIT, "the update pass splits R and G^{-1} into two pieces");
  // the update is skipped under a sticky error (as the CUDA-core update is),
  // before any mbarrier or TMEM exists
  if constexpr (UPDATE)
    if (sticky_error(p.status)) return;
  using C = Cfg<RP, SPLIT, LOSS, SKIPM != 0>;
  constexpr int BN = C::BN, NB = C::NB, NSTAGE = C::NSTAGE, NWB = C::NWB;
  constexpr bool VOTE = SKIPM == 1, RANGE = SKIPM == 2;
  static_assert(SKIPM == 0 || (EPI == 1 && !LOSS), "skipping is a Delta-form option");
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint8_t* stages = smem;
  const uint32_t wsm0 = smem_u32(smem + C::OFF_W);    // W tiles (WSMEM)
  uint64_t* bars = (uint64_t*)(smem + C::OFF_BARS);
  uint32_t* tmem_slot = (uint32_t*)(bars + C::NBAR);
  volatile int* abort_flag = (volatile int*)(tmem_slot + 1);
  double* red = (double*)(smem + C::OFF_BARS + C::NBAR * 8 + 64);
  volatile uint32_t* pflag = (volatile uint32_t*)red;   // [NB][8] (panel kernel; it has no reduction)

  const uint32_t b_full = smem_u32(bars);
  const uint32_t b_empty = b_full + 8 * NSTAGE;
  const uint32_t b_lfull = b_empty + 8 * NSTAGE;
  const uint32_t b_pfull = b_lfull + 8 * NB;
  const uint32_t b_lfree = b_pfull + 8 * NB;
  const uint32_t b_rfull = b_lfree + 8 * NB;
  const uint32_t b_rempty = b_rfull + 16;
  const uint32_t b_wfull = b_rempty + 16;
  const uint32_t b_wempty = b_wfull + 16;
  const uint32_t b_drain = b_wempty + 16;
  const uint32_t b_drain2 = b_drain + 8;

  // (broadcast, so that the compiler knows the roles' branches are uniform and
  // keeps the MMA warp's addresses and descriptors in uniform registers)
  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int i = 0; i < NSTAGE; ++i) {
      mbar_init(b_full + 8 * i, 1);
      mbar_init(b_empty + 8 * i, 1);
    }
    for (int i = 0; i < NB; ++i) {
      mbar_init(b_lfull + 8 * i, 1);
      mbar_init(b_pfull + 8 * i, C::HALF ? 8 : 4);   // the warps of both epilogue warpgroups, or of one
      mbar_init(b_lfree + 8 * i, LOSS ? 4 : 1);      // one warpgroup, or MMA2's commit
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(b_rfull + 8 * i, 1);
      mbar_init(b_rempty + 8 * i, kEpiThreads / 32);
      mbar_init(b_wfull + 8 * i, C::WSMEM ? 1 : kEpiThreads / 32);   // TMA, or the epilogue warps
      mbar_init(b_wempty + 8 * i, 1);
    }
    mbar_init(b_drain, 1);
    mbar_init(b_drain2, 1);
    *abort_flag = 0;
    fence_mbar_init();
  }
  if (warp == kProducerWarp) {
    tmem_alloc(smem_u32(tmem_slot), 512);
    tmem_relinquish();
    if (lane == 0) {
      prefetch_tmap(&tq_hi);
      if (C::NQ > 1) prefetch_tmap(&tq_lo);
      if (C::NQ > 2) prefetch_tmap(&tq_lo2);
      if (C::WSMEM) prefetch_tmap(&tw);
    }
  }
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = *tmem_slot;

  const int64_t ntiles = (p.M + BM - 1) / BM;
  const int64_t kz = blockIdx.z;
  const int64_t kq0 = p.ksplit ? p.q0 + kz * p.ksplit : p.q0;       // this CTA's Q-side rows
  const int64_t kK = p.ksplit ? (p.K - kz * p.ksplit < p.ksplit ? p.K - kz * p.ksplit : p.ksplit) : p.K;
  float* const Rout = p.ksplit ? p.R + kz * p.rstride : p.R;
  const int64_t nchunks = (kK + BN - 1) / BN;
  const int64_t kc0 = (kq0 - p.q0) / BN;   // this CTA's first chunk within the tile's mask

  // The MMAs of one chunk's products (issued by a converged warp).  Descriptors:
  // only the start address varies; WSMEM: the W tile in the same K-major
  // swizzled panels as a chunk.
  // In the Z form of the bf16 mode MMA1 forms -L (its A operand negated), so
  // that the epilogue needs one conversion with a clamp at zero, P = max(0,
  // -L), and MMA2 negates it: -P = min(0, L).
  constexpr bool NEG1 = MODE == 0 && EPI == 0 && !SPLIT;
  const uint64_t dq1 = sdesc(smem_u32(stages), 16, 8 * C::ROWB, C::SWZ);   // a chunk, K-major
  const uint64_t dw = sdesc(wsm0, 16, 8 * C::ROWB, C::SWZ);
  auto mma1 = [&](int st, int lb, int wb) {
    constexpr uint32_t idesc1 = idesc_bf16(BM, BN, false, NEG1);
    const uint32_t wh = tmem + C::COL_W + wb * C::WCOLS, wl = wh + RP / 2;
    const uint32_t bo = (uint32_t)st * (C::STAGE_BYTES >> 4), ao = (uint32_t)wb * (C::W_BYTES >> 4);
    const uint32_t d = tmem + C::COL_L + lb * BN;
#pragma unroll
    for (int k = 0; k < RP / 16; ++k) {
      constexpr int PW = C::PANEL_W;
      const uint32_t off = bo + (((k * 16 / PW) * C::PANEL_BYTES + ((k * 16) % PW) * 2) >> 4);
      const uint32_t aoff = ao + (((k * 16 / PW) * C::W_PANEL_BYTES + ((k * 16) % PW) * 2) >> 4);
      if (C::WSMEM) mma_ss_elect(d, dw, aoff, dq1, off, idesc1, k > 0);
      else mma_ts_elect(d, wh + k * 8, dq1, off, idesc1, k > 0);
      if (SPLIT) {
        mma_ts_elect(d, wh + k * 8, dq1, off + (C::OPER_BYTES >> 4), idesc1, 1);
        mma_ts_elect(d, wl + k * 8, dq1, off, idesc1, 1);
      }
    }
  };
  // R columns [hcol, hcol + NR) of Q: their panels start hcol / PANEL_W panels in
  const uint32_t hpan = C::RHALF ? (uint32_t)blockIdx.y * (C::NR / C::PANEL_W) * C::PANEL_BYTES : 0u;
  const uint64_t dq2 = sdesc(smem_u32(stages) + hpan, C::PANEL_BYTES, 8 * C::ROWB, C::SWZ);   // a chunk, MN-major
  auto mma2 = [&](int st, int lb, int rb, bool accumulate) {
    constexpr uint32_t idesc2 = idesc_bf16(BM, LOSS ? 16 : C::NR, true, !SPLIT);
    const uint32_t bo = (uint32_t)st * (C::STAGE_BYTES >> 4);
    const uint32_t pl = tmem + C::COL_L + lb * BN;
    const uint32_t dr = tmem + C::COL_R + rb * C::RCOLS;
#pragma unroll
    for (int k = 0; k < BN / 16; ++k) {
      const uint32_t off = bo + ((k * 16 * C::ROWB) >> 4);
      const uint32_t acc = k > 0 || accumulate ? 1u : 0u;
      if (!SPLIT) {             // P q_hi; each warpgroup's P starts at its own columns of L
        constexpr int KH = BN / 32;   // k steps per half
        mma_ts_elect(dr, pl + (C::HALF ? (k / KH) * (BN / 2) + (k % KH) * 8 : k * 8), dq2, off, idesc2, acc);
      } else {                  // P_hi (q_hi + q_lo + q_lo2) + P_lo q_hi
        const uint32_t ph = pl + (k / 2) * 32 + (k % 2) * 8, plo = ph + 16;
        mma_ts_elect(dr, ph, dq2, off, idesc2, acc);
        mma_ts_elect(dr, ph, dq2, off + (C::OPER_BYTES >> 4), idesc2, 1);
        mma_ts_elect(dr, ph, dq2, off + ((2 * C::OPER_BYTES) >> 4), idesc2, 1);
        mma_ts_elect(dr, plo, dq2, off, idesc2, 1);
      }
    }
  };
  // Delta form: a chunk whose P is zero in every row adds nothing to R (Sec.
  // 4.3); its MMAs are skipped, except for the first chunk of a tile, which
  // initialises the accumulator
  auto vanishes = [&](int lb, bool first) -> bool {
    if (!VOTE || first) return false;
    uint32_t nz = 0u;
#pragma unroll
    for (int w = 0; w < (C::HALF ? 8 : 4); ++w) nz |= pflag[8 * lb + w];
    if (nz == 0u && p.skips != nullptr && lane == 0) atomicAdd(p.skips, 1ull);
    return nz == 0u;
  };

  if (warp == kProducerWarp) {
    // ------------------------------------------------------------ producer
    if (lane == 0) {
      int64_t G = 0, tt = 0;
      bool ok = true;
      for (int64_t t = blockIdx.x; t < ntiles && ok; t += gridDim.x, ++tt) {
        if (C::WSMEM) {   // the tile's W rows into W buffer tt % NWB once MMA1 is done with it
          const int wb = (int)(tt % NWB);
          if (!(ok = wait_bar(b_wempty + 8 * wb, (uint32_t)((tt / NWB) & 1) ^ 1u, abort_flag, p.status, 10)))
            break;
          mbar_expect_tx(b_wfull + 8 * wb, C::W_BYTES);
#pragma unroll
          for (int pn = 0; pn < C::NPANEL; ++pn)
            tma_load_2d(wsm0 + wb * C::W_BYTES + pn * C::W_PANEL_BYTES, &tw, b_wfull + 8 * wb, pn * C::PANEL_W,
                        (int)(p.m0 + t * BM));
        }
        int64_t clast, nlive;
        const ChunkMask cm = chunk_mask<RANGE>(p, t, kc0, nchunks, &clast, &nlive);
        for (int64_t c = 0; c < nchunks; ++c) {
          if (RANGE && !cm.live(c)) continue;
          const int s = (int)(G % NSTAGE);
          if (!(ok = wait_bar(b_empty + 8 * s, (uint32_t)((G / NSTAGE) & 1) ^ 1u, abort_flag, p.status, 1)))
            break;
          mbar_expect_tx(b_full + 8 * s, C::STAGE_BYTES);
          const uint32_t dst = smem_u32(stages + (size_t)s * C::STAGE_BYTES);
          const int y = (int)(kq0 + c * BN);
#pragma unroll
          for (int pn = 0; pn < C::NPANEL; ++pn) {
            tma_load_2d(dst + pn * C::PANEL_BYTES, &tq_hi, b_full + 8 * s, pn * C::PANEL_W, y);
            if (C::NQ > 1)
              tma_load_2d(dst + C::OPER_BYTES + pn * C::PANEL_BYTES, &tq_lo, b_full + 8 * s, pn * C::PANEL_W, y);
            if (C::NQ > 2)
              tma_load_2d(dst + 2 * C::OPER_BYTES + pn * C::PANEL_BYTES, &tq_lo2, b_full + 8 * s, pn * C::PANEL_W,
                          y);
          }
          ++G;
        }
      }
      if (!ok) {  // drain the copies still in flight before shared memory goes away
        for (int64_t k = G - NSTAGE > 0 ? G - NSTAGE : 0; k < G; ++k) {
          uint64_t t0 = globaltimer_ns();
          while (!mbar_try_wait(b_full + 8 * (int)(k % NSTAGE), (uint32_t)((k / NSTAGE) & 1)) &&
                 globaltimer_ns() - t0 < 100000000ull) {
          }
        }
        // W loads: those of tiles [0, tt) were issued, only the last NWB can
        // still be in flight
        for (int64_t k = tt - NWB > 0 ? tt - NWB : 0; C::WSMEM && k < tt; ++k) {
          uint64_t t0 = globaltimer_ns();
          while (!mbar_try_wait(b_wfull + 8 * (int)(k % NWB), (uint32_t)((k / NWB) & 1)) &&
                 globaltimer_ns() - t0 < 100000000ull) {
          }
        }
      }
    }
  } else if (warp == kMma1Warp) {
    // ------------------------------------------------------------ MMA1 issuer
    // L[lb] = W tile x chunk^T for every chunk of this CTA's tiles, in order.
    // L[lb] may be overwritten once the second product has read P from it, which
    // its commit on b_lfree says: products into different accumulators have no
    // order of their own.
    int s1 = 0, l1 = 0, wb1 = 0;
    uint32_t ph_full = 0, ph_lfree = 1, ph_wfull = 0;
    ChunkWalk<RANGE> k1(p, (int)ntiles, (int)nchunks, kc0);
    auto advance1 = [&](bool last) {
      s1 = s1 == NSTAGE - 1 ? 0 : s1 + 1;
      ph_full ^= s1 == 0 ? 1u : 0u;
      l1 = l1 == NB - 1 ? 0 : l1 + 1;
      ph_lfree ^= l1 == 0 ? 1u : 0u;
      if (NWB == 2) wb1 ^= last ? 1 : 0;
      ph_wfull ^= (last && wb1 == 0) ? 1u : 0u;
      k1.next(p);
    };
    // A chunk's barriers are tested while the chunk before is issued; with a
    // range-search mask, whose words past the 64th chunk come from global memory,
    // only where the products are short (exact sweeps, ahead / not: 139,255 rows at r = 64
    // in the bf16 mode 15.1 / 15.4 ms; 60,000 rows at r = 100 in the fp32-accurate mode
    // 12.36 / 11.26 ms, 40,000 at r = 200 in the bf16 mode 4.49 / 4.11 ms).
    constexpr bool AHEAD = !RANGE || (!SPLIT && RP <= 128);
    bool ready = false;
    while (k1.valid()) {
      if (!ready && (!conv_wait(b_full + 8 * s1, ph_full, abort_flag, p.status, 3) ||
                     !conv_wait(b_lfree + 8 * l1, ph_lfree, abort_flag, p.status, 4)))
        break;
      if (k1.first) {
        if (!conv_wait(b_wfull + 8 * wb1, ph_wfull, abort_flag, p.status, 2)) break;
        if (RANGE && p.skips != nullptr && lane == 0 && k1.nlive < k1.n)
          atomicAdd(p.skips, (unsigned long long)(k1.n - k1.nlive));
      }
      fence_after();
      const bool last = k1.last();
      const int s = s1, l = l1, wb = wb1;
      bool next = false;
      if (AHEAD) {
        advance1(last);
        next = mbar_test_wait(b_full + 8 * s1, ph_full) & mbar_test_wait(b_lfree + 8 * l1, ph_lfree);
      }
      mma1(s, l, wb);
      commit_elect(b_lfull + 8 * l);
      if (LOSS) commit_elect(b_empty + 8 * s);
      if (last) commit_elect(b_wempty + 8 * wb);
      if (AHEAD) ready = __all_sync(0xffffffffu, next);
      else advance1(last);
    }
    // wait until every MMA issued by this warp has completed
    commit_elect(b_drain);
    if (lane == 0) {
      const uint64_t t0 = globaltimer_ns();
      while (!mbar_try_wait(b_drain, 0) && globaltimer_ns() - t0 < 200000000ull) {
      }
    }
    __syncwarp();
  } else if (warp == kMma2Warp) {
    // ------------------------------------------------------------ MMA2 issuer
    // R += P[lb] x chunk for every chunk once its P is in TMEM; frees the
    // shared-memory stage and the L buffer, and hands R over per tile.
    if constexpr (!LOSS) {
      int s2 = 0, l2 = 0, rb2 = 0;
      uint32_t ph_pfull = 0, ph_rempty = 1;
      ChunkWalk<RANGE> k2(p, (int)ntiles, (int)nchunks, kc0);
      while (k2.valid()) {
        // (a first test that may suspend the thread where the wait is long: fp32-
        // accurate, r_pad = 256: 1,366 -> 1,335 us, 40,000 rows against 8,192; bf16: 257
        // -> 263 us, with vote skipping 1,372 -> 1,381 us)
        constexpr bool LONG = SPLIT && RP == 256 && SKIPM == 0;
        const bool here = LONG ? mbar_try_wait(b_pfull + 8 * l2, ph_pfull) : mbar_test_wait(b_pfull + 8 * l2, ph_pfull);
        if (!conv_wait(here, b_pfull + 8 * l2, ph_pfull, abort_flag, p.status, 5)) break;
        if (k2.first && !conv_wait(b_rempty + 8 * rb2, ph_rempty, abort_flag, p.status, 6)) break;
        fence_after();
        const bool last = k2.last();
        if (!vanishes(l2, k2.first)) mma2(s2, l2, rb2, !k2.first);
        commit_elect(b_lfree + 8 * l2);
        commit_elect(b_empty + 8 * s2);
        if (last) commit_elect(b_rfull + 8 * rb2);
        s2 = s2 == NSTAGE - 1 ? 0 : s2 + 1;
        l2 = l2 == NB - 1 ? 0 : l2 + 1;
        ph_pfull ^= l2 == 0 ? 1u : 0u;
        if (C::NRB == 2) rb2 ^= last ? 1 : 0;
        ph_rempty ^= (last && rb2 == 0) ? 1u : 0u;
        k2.next(p);
      }
      commit_elect(b_drain2);
      if (lane == 0) {
        const uint64_t t0 = globaltimer_ns();
        while (!mbar_try_wait(b_drain2, 0) && globaltimer_ns() - t0 < 200000000ull) {
        }
      }
      __syncwarp();
    }
  } else {
    // ------------------------------------------------------------ epilogue
    // Two warpgroups take alternate chunks (HALF: half of every chunk's
    // columns each); within a warpgroup thread t owns TMEM lane t = tile row
    // t.  Tile-level work (W load, R readout) is split by columns between the
    // two warpgroups.
    const int wg = warp >> 2;
    const int row = (warp & 3) * 32 + lane;
    const int et = threadIdx.x;                          // 0 .. 255
    const uint32_t lane_base = ((uint32_t)((warp & 3) * 32)) << 16;
    // (loss) the chunks' sums of a row, as an fp32 sum and its rounding errors
    // (exact but for the errors' own sum, 2^-48); fp64 adds, two a chunk and
    // thread, cost more than the pass's tensor work.  Per tile into fp64, and
    // before that where the fp32 sums would leave their range (see below).
    double s2 = 0.0, s1 = 0.0;
    float h2 = 0.f, l2 = 0.f, h1 = 0.f, l1 = 0.f;
    auto two_sum = [](float& h, float& l, float x) {
      const float t = h + x, z = t - h;
      l += (h - (t - z)) + (x - z);
      h = t;
    };
    float nbest = -INFINITY;   // nearest-neighbour pass: this thread's best L of its row so far
    int64_t nidx = -1;
    bool ok = true;
    // loss pass: this thread's row of S, walked alongside the column chunks so
    // that support entries are left to the support pass (no cancellation)
    constexpr int kWin = 32;
    int64_t se = 0, send = 0;              // the row's entries from the window's first to its last
    int wpos = 0, wcnt = 0;                // position in the window, entries in it
    int64_t snext = INT_MAX;               // the next entry's column (see support_mask)
    int* win = (int*)(smem + C::OFF_WIN) + et * (kWin + 1);

    // load the W tile `tile` into W buffer wb: warpgroup g takes 8-word groups g, g+2, ...
    auto load_w = [&](int64_t tile, int wb) {
      if constexpr (C::WSMEM) return;   // loaded by the producer's TMA
      const int64_t li = tile * BM + row;
      const bool valid = li < p.M;
      if constexpr (UPDATE) {
        // R + Rs of this row, split into hi = bf16(x) and lo = bf16(x - hi)
        const float* src = p.upd_R + (valid ? li : 0) * RP;
        const float* srs = p.upd_Rs + (valid ? li : 0) * RP;
        const bool flg = valid && p.upd_flags[li] != 0;
        const uint32_t wcol = tmem + lane_base + C::COL_W + wb * C::WCOLS;
#pragma unroll 1
        for (int q = wg; q < RP / 16; q += 2) {
          float x[16];
#pragma unroll
          for (int k = 0; k < 16; k += 4) {
            float4 a = valid ? __ldg((const float4*)(src + 16 * q + k)) : make_float4(0.f, 0.f, 0.f, 0.f);
            if (flg) {
              const float4 b = __ldg((const float4*)(srs + 16 * q + k));
              a.x += b.x; a.y += b.y; a.z += b.z; a.w += b.w;
            }
            x[k] = a.x; x[k + 1] = a.y; x[k + 2] = a.z; x[k + 3] = a.w;
          }
          uint32_t vh[8], vl[8];
#pragma unroll
          for (int k = 0; k < 8; ++k) {
            const uint32_t h = pack_bf16x2(x[2 * k], x[2 * k + 1]);
            vh[k] = h;
            vl[k] = pack_bf16x2(x[2 * k] - __uint_as_float(h << 16), x[2 * k + 1] - __uint_as_float(h & 0xffff0000u));
          }
          tmem_st8(wcol + q * 8, vh);
          tmem_st8(wcol + RP / 2 + q * 8, vl);
        }
        tmem_wait_st();
        fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(b_wfull + 8 * wb);
        return;
      }
      const uint4* src = (const uint4*)(p.Mhi + (p.m0 + (valid ? li : 0)) * RP);
      const uint4* srcl = (const uint4*)(p.Mlo + (p.m0 + (valid ? li : 0)) * RP);
      const uint32_t wcol = tmem + lane_base + C::COL_W + wb * C::WCOLS;
#pragma unroll
      for (int q = wg; q < RP / 16; q += 2) {
        uint4 a = valid ? __ldg(src + 2 * q) : make_uint4(0, 0, 0, 0);
        uint4 b = valid ? __ldg(src + 2 * q + 1) : make_uint4(0, 0, 0, 0);
        uint32_t v[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
        tmem_st8(wcol + q * 8, v);
        if (SPLIT) {
          uint4 c = valid ? __ldg(srcl + 2 * q) : make_uint4(0, 0, 0, 0);
          uint4 e = valid ? __ldg(srcl + 2 * q + 1) : make_uint4(0, 0, 0, 0);
          uint32_t w[8] = {c.x, c.y, c.z, c.w, e.x, e.y, e.z, e.w};
          tmem_st8(wcol + RP / 2 + q * 8, w);
        }
      }
      tmem_wait_st();
      fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(b_wfull + 8 * wb);
    };

    // Loss pass: this row's entries in columns [c0, c0 + BN) as bits (bit b of
    // m0: column c0 + b, of m1: c0 + 64 + b), c0 ascending within a tile.  The
    // row's next entries sit in a window of kWin column indices in shared memory
    // (a dependent global load per entry held the epilogue up for most of the
    // pass), refilled by the row's own thread, its loads in flight together; the
    // next column is kept in a register, so that a warp without an entry in the
    // chunk passes on after one vote.  Where few rows need more entries than
    // their windows hold, the whole warp reads on in each, 256 entries at a time;
    // a row with many entries per chunk (a hub of the graph has one in every
    // column) is left without a window and read that way in every chunk.
    // Called by converged warps.
    auto refill = [&](int64_t from) {   // this thread's window: entries [from, from + kWin) of its row
      se = from;
      wpos = 0;
      wcnt = (int)(send - from < kWin ? send - from : kWin);
      for (int h = 0; h < wcnt; h += 16) {
        int col[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) col[i] = h + i < wcnt ? p.cidx[from + h + i] : 0;
#pragma unroll
        for (int i = 0; i < 16; ++i) win[h + i] = col[i];
      }
      snext = wcnt > 0 ? win[0] : INT_MAX;
    };
    auto set_bit = [](uint64_t& m0, uint64_t& m1, int b) {
      const uint64_t bit = 1ull << (b & 63);
      m0 |= b < 64 ? bit : 0ull;
      m1 |= b < 64 ? 0ull : bit;
    };
    auto support_mask = [&](int64_t c0, uint64_t& m0, uint64_t& m1) {
      m0 = m1 = 0ull;
      const int64_t cend = c0 + BN;
      // snext: the next column; INT_MIN: more entries, not in the window; INT_MAX: none
      while (__any_sync(0xffffffffu, snext < cend)) {
        while (snext < cend && snext != INT_MIN) {
          const int b = (int)(snext - c0);
          if (b >= 0) set_bit(m0, m1, b);
          ++wpos;
          snext = wpos < wcnt ? win[wpos] : se + wcnt < send ? INT_MIN : INT_MAX;
        }
        __syncwarp();
        uint32_t more = __ballot_sync(0xffffffffu, snext == INT_MIN);
        if (__popc(more) > 4) {
          if (snext == INT_MIN) refill(se + wcnt);
          __syncwarp();
          continue;
        }
        while (more) {
          const int src = __ffs(more) - 1;
          more &= more - 1;
          int64_t q = __shfl_sync(0xffffffffu, se + wcnt, src);
          const int64_t e = __shfl_sync(0xffffffffu, send, src), q0 = q;
          uint64_t a0 = 0ull, a1 = 0ull;
          int n;
          do {
            int col[8];
#pragma unroll
            for (int k = 0; k < 8; ++k) col[k] = q + lane + 32 * k < e ? p.cidx[q + lane + 32 * k] : INT_MAX;
            n = 0;
#pragma unroll
            for (int k = 0; k < 8; ++k) {
              const bool in = col[k] < cend;   // (columns lie below INT_MAX)
              n += __popc(__ballot_sync(0xffffffffu, in && col[k] != INT_MAX));
              if (in && col[k] != INT_MAX && col[k] >= c0) set_bit(a0, a1, (int)(col[k] - c0));
            }
            q += n;
          } while (n == 256);
#pragma unroll
          for (int w = 0; w < 2; ++w) {
            const uint64_t a = w ? a1 : a0;
            const uint64_t all = ((uint64_t)__reduce_or_sync(0xffffffffu, (uint32_t)(a >> 32)) << 32) |
                                 __reduce_or_sync(0xffffffffu, (uint32_t)a);
            if (lane == src) {
              if (w) m1 |= all;
              else m0 |= all;
            }
          }
          if (lane == src) {
            if (q - q0 >= 16 && q < e) {   // no window: the warp reads on in the next chunk
              se = q;
              wpos = wcnt = 0;
              snext = INT_MIN;
            } else {
              refill(q);
            }
          }
          __syncwarp();
        }
        break;   // those rows go on past the chunk, or end
      }
    };

    // R of a tile, the n-th of this CTA
    auto readout = [&](int tile, int n) -> bool {
      const int rb = n % C::NRB;
      if (!conv_wait(b_rfull + 8 * rb, (uint32_t)((n / C::NRB) & 1), abort_flag, p.status, 8)) return false;
      fence_after();
      const int64_t li0 = (int64_t)tile * BM + (warp & 3) * 32;
      if constexpr (MODE == 0)
        store_r_tile<C::NR, RP>(tmem + lane_base + C::COL_R + rb * C::RCOLS, b_rempty + 8 * rb,
                                (float*)(smem + C::OFF_STG) + warp * 1024,
                                Rout + li0 * RP + (C::RHALF ? (int64_t)blockIdx.y * C::NR : 0), li0, p.M, wg, lane);
      return true;
    };

    {  // prologue: the first NWB tiles
      int tt = 0;
      for (int t = blockIdx.x; t < (int)ntiles && tt < NWB; t += gridDim.x, ++tt) load_w(t, tt);
    }
    int tt = 0;          // tiles this CTA has processed
    int lb = NB - 1;     // L buffer of the current chunk and the parity of its use
    uint32_t lpar = 1;
    bool odd = true;     // the chunks alternate between the warpgroups
    int pend = -1;       // a tile whose R is still to be read out (NRB = 2)
    for (int t = blockIdx.x; t < (int)ntiles && ok; t += gridDim.x, ++tt) {
      int64_t clast, nlive;
      const ChunkMask cm = chunk_mask<RANGE>(p, t, kc0, nchunks, &clast, &nlive);
      if (SUMS) {
        const int64_t li = (int64_t)t * BM + row;
        send = li < p.M ? p.rowptr[li + 1] : 0;
        refill(li < p.M ? p.rowptr[li] : 0);
      }
      for (int ci = 0; ci < (int)nchunks; ++ci) {
        if (RANGE && !cm.live(ci)) continue;
        const int64_t c = ci;
        if (++lb == NB) { lb = 0; lpar ^= 1u; }
        odd = !odd;
        if (!C::HALF && odd != (wg != 0)) continue;
        // the support columns of this chunk, one bit each, found while the
        // chunk's product is under way
        uint64_t m0 = 0ull, m1 = 0ull;
        if (SUMS) support_mask(c * BN, m0, m1);
        if (!(ok = conv_wait(b_lfull + 8 * lb, lpar, abort_flag, p.status, 7))) break;
        fence_after();
        const int kv = (int)(kK - c * BN < BN ? kK - c * BN : BN);   // valid columns in this chunk
        const uint32_t lcol = tmem + lane_base + C::COL_L + lb * BN;
        float2 c2a = make_float2(0.f, 0.f), c2b = c2a, c1 = c2a;   // (loss) sums of relu(x)^2 and of relu(x)
        uint32_t nzacc = 0u;   // Delta form: OR of this thread's P words
        // MODE 0: P of one group of 32 columns of L (TMEM columns [32 g, 32 g + 32)
        // of the buffer): bf16, 16 TMEM columns at 16 g (HALF: within the
        // warpgroup's own half of the buffer); fp32-accurate: hi and lo, 32 at 32
        // g.  P never overwrites L columns that are still to be read.
        auto to_p = [&](const uint32_t(&v)[32], int g) {
          if (!SPLIT) {
            // max(0, L) (Delta form) or max(0, -L) (Z form, v holds -L); MMA2
            // negates both.  A NaN stays a NaN.
            uint32_t pk[16];
#pragma unroll
            for (int i = 0; i < 16; ++i) {
              pk[i] = pack_relu_bf16x2(__uint_as_float(v[2 * i]), __uint_as_float(v[2 * i + 1]));
              if (VOTE) nzacc |= pk[i] & 0x7fff7fffu;   // -0 counts as zero
            }
            tmem_st16(C::HALF ? lcol + wg * (BN / 2) + (g - wg * (BN / 64)) * 16 : lcol + g * 16, pk);
          } else {
            // fp32-accurate: P = hi + lo, hi at columns [32 g, 32 g + 16), lo at [32 g + 16, 32 g + 32)
            uint32_t ph[16], pl[16];
#pragma unroll
            for (int i = 0; i < 16; ++i) {
              const float x0 = __uint_as_float(v[2 * i]), x1 = __uint_as_float(v[2 * i + 1]);
              const float e0 = EPI == 0 ? fminf(0.f, x0) : fminf(0.f, -x0);
              const float e1 = EPI == 0 ? fminf(0.f, x1) : fminf(0.f, -x1);
              const uint32_t hp = pack_bf16x2(e0, e1);
              const float h0 = __uint_as_float(hp << 16), h1 = __uint_as_float(hp & 0xffff0000u);
              ph[i] = hp;
              pl[i] = pack_bf16x2(e0 - h0, e1 - h1);
              if (VOTE) nzacc |= (ph[i] | pl[i]) & 0x7fff7fffu;   // -0 counts as zero
            }
            tmem_st16(lcol + g * 32, ph);
            tmem_st16(lcol + g * 32 + 16, pl);
          }
        };
        // the first-product passes: one group of 32 columns, columns past the
        // Q side masked
        auto group = [&](uint32_t(&v)[32], int g) {
          if (!NEAREST && kv < BN) {
#pragma unroll
            for (int i = 0; i < 32; ++i)
              if (g * 32 + i >= kv) v[i] = 0u;
          }
          if (UPDATE) {   // X for columns [col0, col0 + 32) of this row: the step
            const int64_t li = (int64_t)t * BM + row;
            if (li < p.M) {
              const int64_t col0 = c * BN + g * 32;
              float* mrow = p.upd_M + (p.upd_row0 + li) * RP + col0;
              float* erow = p.upd_E + (p.upd_row0 + li) * RP + col0;
              uint32_t hw[16];
              bool finite = true;
#pragma unroll
              for (int k = 0; k < 32; k += 4) {
                const float4 mo = *(const float4*)(mrow + k);
                const float4 eo = p.momentum ? *(const float4*)(erow + k) : make_float4(0.f, 0.f, 0.f, 0.f);
                const float mv[4] = {mo.x, mo.y, mo.z, mo.w}, evo[4] = {eo.x, eo.y, eo.z, eo.w};
                float nv[4], ev[4];
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                  const float x = __uint_as_float(v[k + j]);
                  const float u = p.delta_form ? p.eta * x : p.eta * (x - mv[j]);
                  ev[j] = p.momentum ? fmaf(p.gamma, evo[j], u) : u;
                  nv[j] = mv[j] + ev[j];
                  finite = finite && isfinite(nv[j]);
                }
                *(float4*)(mrow + k) = make_float4(nv[0], nv[1], nv[2], nv[3]);
                if (p.momentum) *(float4*)(erow + k) = make_float4(ev[0], ev[1], ev[2], ev[3]);
                hw[k / 2] = pack_bf16x2(nv[0], nv[1]);
                hw[k / 2 + 1] = pack_bf16x2(nv[2], nv[3]);
              }
              uint4* hrow = (uint4*)(p.upd_hi + (p.upd_row0 + li) * RP + col0);
#pragma unroll
              for (int k = 0; k < 4; ++k) hrow[k] = make_uint4(hw[4 * k], hw[4 * k + 1], hw[4 * k + 2], hw[4 * k + 3]);
              if (!finite) record(p.status, NMD_ERR_DIVERGED, (int)(p.upd_row0 + li));
            }
          } else if (NEAREST) {
            // columns past the set or the row itself do not count; the group's
            // largest value first, its (first) place only where it beats the
            // row's best so far
            const int64_t cb = c * BN + g * 32, self = (int64_t)t * BM + row;
            if (kv < BN || (self >= cb && self < cb + 32)) {
#pragma unroll
              for (int i = 0; i < 32; ++i)
                if (g * 32 + i >= kv || cb + i == self) v[i] = 0xff800000u;   // -inf
            }
            float gm = __uint_as_float(v[0]);
#pragma unroll
            for (int i = 1; i < 32; ++i) gm = fmaxf(gm, __uint_as_float(v[i]));
            if (gm > nbest) {
              // the places of that value as bits.  Nearly every group of a row's
              // first chunks comes here, which are all there is of a small set:
              // 3,000 rows take 18 us, 46 with a selection of value and 64-bit
              // index per column (30,000 rows of up to 16 columns: 260, 465)
              uint32_t at = 0u, neg = 0u;
#pragma unroll
              for (int i = 0; i < 32; ++i) at |= __uint_as_float(v[i]) == gm ? 1u << i : 0u;
              const int first = __ffs(at) - 1;
              nbest = gm;
              nidx = cb + first;
              if (gm == 0.f) {   // of zeros, too, the first one's sign
#pragma unroll
                for (int i = 0; i < 32; ++i) neg |= (v[i] >> 31) << i;
                nbest = (neg >> first) & 1u ? -0.f : 0.f;
              }
            }
          } else if (SUMS) {
            const uint32_t mg = (uint32_t)((g < 2 ? m0 : m1) >> (32 * (g & 1)));
            if (__any_sync(0xffffffffu, mg != 0u)) {   // support columns in this group: zero them
#pragma unroll
              for (int i = 0; i < 32; ++i)
                if ((mg >> i) & 1u) v[i] = 0u;
            }
            // pairs of columns in packed FMAs, in two chains: one fp32 chain of
            // 128 dependent FMAs a chunk set the pace of this loop
#pragma unroll
            for (int i = 0; i < 32; i += 4) {
              const float2 ta = make_float2(fmaxf(0.f, __uint_as_float(v[i])), fmaxf(0.f, __uint_as_float(v[i + 1])));
              const float2 tb = make_float2(fmaxf(0.f, __uint_as_float(v[i + 2])), fmaxf(0.f, __uint_as_float(v[i + 3])));
              c2a = ffma2(ta, ta, c2a);
              c2b = ffma2(tb, tb, c2b);
              c1 = fadd2(c1, fadd2(ta, tb));
            }
          }
        };
        if constexpr (MODE == 0) {
          constexpr int NG = C::HALF ? BN / 64 : BN / 32;   // this warpgroup's groups of 32 columns
          const int g0 = C::HALF ? wg * NG : 0;
          uint32_t va[32], vb[32];
          if (kv < BN || p.Lout != nullptr) {
            // a ragged last chunk (columns past the block contribute nothing),
            // or L itself is wanted (tested once a group: a test per column cost
            // 36.6 instead of 32.8 us at r_pad = 16, 139,255 rows against 1,393)
#pragma unroll 1
            for (int g = g0; g < g0 + NG; ++g) {
              tmem_ld32(lcol + g * 32, va);
              tmem_wait_ld(va);
              const int64_t li = (int64_t)t * BM + row;
              const int n = kv - g * 32;   // valid columns of this group
              if (n < 32) {
#pragma unroll
                for (int i = 0; i < 32; ++i) va[i] = i < n ? va[i] : 0u;
              }
              if (p.Lout != nullptr && li < p.M) {   // (the bf16 mode's Z form holds -L)
                float* lrow = p.Lout + li * p.K + c * BN + g * 32;
#pragma unroll
                for (int i = 0; i < 32; ++i)
                  if (i < n) lrow[i] = EPI == 0 && !SPLIT ? -__uint_as_float(va[i]) : __uint_as_float(va[i]);
              }
              to_p(va, g);
            }
          } else {
            // the next group's load in flight while one is converted
            tmem_ld32(lcol + g0 * 32, va);
#pragma unroll
            for (int q = 0; q < NG; q += 2) {
              tmem_wait_ld(va);
              if (q + 1 < NG) tmem_ld32(lcol + (g0 + q + 1) * 32, vb);
              to_p(va, g0 + q);
              if (q + 1 < NG) {
                tmem_wait_ld(vb);
                if (q + 2 < NG) tmem_ld32(lcol + (g0 + q + 2) * 32, va);
                to_p(vb, g0 + q + 1);
              }
            }
          }
        } else {
          // groups of 32 columns, the next one's load in flight while one is taken
          uint32_t va[32], vb[32];
          tmem_ld32(lcol, va);
#pragma unroll 1
          for (int q = 0; q < BN / 32; q += 2) {
            tmem_wait_ld(va);
            tmem_ld32(lcol + q * 32 + 32, vb);
            group(va, q);
            tmem_wait_ld(vb);
            if (q + 2 < BN / 32) tmem_ld32(lcol + q * 32 + 64, va);
            group(vb, q + 1);
          }
        }
        if (LOSS) {
          if (SUMS) {
            const float x2 = (c2a.x + c2b.x) + (c2a.y + c2b.y), x1 = c1.x + c1.y;
            // a chunk's sum of squares is finite while L is below about 2e18, a
            // row's sum of such chunks need not be: into fp64 in time (an
            // infinite chunk, too, whose error term would not be a number).  The
            // plain sums, by Cauchy's inequality the smaller ones, go with them.
            if (__any_sync(0xffffffffu, h2 + x2 > 1e38f)) {
              s2 += (double)h2 + (double)l2 + (double)x2;
              s1 += (double)h1 + (double)l1 + (double)x1;
              h2 = l2 = h1 = l1 = 0.f;
            } else {
              two_sum(h2, l2, x2);
              two_sum(h1, l1, x1);
            }
          }
          fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(b_lfree + 8 * lb);
        } else {
          if (VOTE) {   // published before the arrive (release) that MMA2 acquires
            const bool nz = __any_sync(0xffffffffu, nzacc != 0u);
            if (lane == 0) pflag[8 * lb + (C::HALF ? warp : (warp & 3))] = nz ? 1u : 0u;
          }
          tmem_wait_st();
          fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(b_pfull + 8 * lb);
          // the previous tile's R, after this warpgroup's first chunk of the tile
          if (C::NRB == 2 && pend >= 0) {
            if (!(ok = readout(pend, tt - 1))) break;
            pend = -1;
          }
        }
      }
      if (!ok) break;
      if (SUMS) {
        s2 += (double)h2 + (double)l2;
        s1 += (double)h1 + (double)l1;
        h2 = l2 = h1 = l1 = 0.f;
      }
      if (NEAREST) {   // this warpgroup's best of the row; the two are merged by atomicMax
        const int64_t li = (int64_t)t * BM + row;
        if (li < p.M && nidx >= 0) {
          const uint32_t b = __float_as_uint(nbest);
          const uint32_t ord = (b & 0x80000000u) ? ~b : (b | 0x80000000u);   // float order as unsigned
          atomicMax(p.nn_key + li, ((unsigned long long)ord << 32) | (unsigned long long)(~(uint32_t)nidx));
        }
        nbest = -INFINITY;
        nidx = -1;
      }
      // refill this tile's W buffer with the tile NWB steps ahead
      const int tn = t + NWB * (int)gridDim.x;
      if (!C::WSMEM && tn < (int)ntiles) {
        const int wb = tt % NWB;
        if (!(ok = conv_wait(b_wempty + 8 * wb, (uint32_t)((tt / NWB) & 1), abort_flag, p.status, 9))) break;
        fence_after();
        load_w(tn, wb);
      }
      if (!LOSS) {
        // (a tile in which this warpgroup had no chunk has not read the previous R yet)
        if (C::NRB == 2 && pend >= 0 && !(ok = readout(pend, tt - 1))) break;
        if (C::NRB == 2) pend = t;
        else if (!(ok = readout(t, tt))) break;
      }
    }
    if (!LOSS && C::NRB == 2 && ok && pend >= 0) readout(pend, tt - 1);
    if (SUMS) {
      // fixed-order reduction over the 256 epilogue threads
      red[2 * et] = s2;
      red[2 * et + 1] = s1;
      named_bar_sync(1, kEpiThreads);
      if (et == 0) {
        double a = 0.0, b = 0.0;
        for (int i = 0; i < kEpiThreads; ++i) {
          a += red[2 * i];
          b += red[2 * i + 1];
        }
        p.parts[(size_t)blockIdx.x * 8 + 0] = a;
        p.parts[(size_t)blockIdx.x * 8 + 1] = b;
      }
    }
  }
  fence_before();
  __syncthreads();
  fence_after();
  if (warp == kProducerWarp) tmem_dealloc(tmem, 512);
}

// Self-test of the bounded wait used by every pipeline wait above: thread 0
// waits on a barrier that nothing arrives at; after limit_ns the wait gives
// up, sets the abort flag and records NMD_ERR_TIMEOUT (detail 99) in the
// status words, and the kernel returns normally.
__global__ void wait_selftest_kernel(int* status, uint64_t limit_ns) {
  __shared__ __align__(8) uint64_t bar;
  __shared__ int abort_flag;
  if (threadIdx.x == 0) {
    mbar_init(smem_u32(&bar), 1);
    abort_flag = 0;
    fence_mbar_init();
  }
  __syncthreads();
  if (threadIdx.x == 0) wait_bar_slow(smem_u32(&bar), 0, &abort_flag, status, 99, limit_ns);
  __syncthreads();
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = (PFN_cuTensorMapEncodeTiled_v12000)p;
  });
  return fn;
}

// Tensor map of a row-major rows x rp bf16 factor copy, box = panel_w x bn.
bool tensor_map(const bf16* base, int64_t rows, int rp, int panel_w, int bn, CUtensorMap* out) {
  static std::mutex mu;
  static std::map<std::tuple<const void*, int64_t, int, int>, CUtensorMap> cache;
  std::lock_guard<std::mutex> g(mu);
  auto key = std::make_tuple((const void*)base, rows, rp, bn);
  auto it = cache.find(key);
  if (it != cache.end()) {
    *out = it->second;
    return true;
  }
  PFN_cuTensorMapEncodeTiled_v12000 fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[2] = {(cuuint64_t)rp, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)rp * 2};
  cuuint32_t box[2] = {(cuuint32_t)panel_w, (cuuint32_t)bn};
  cuuint32_t es[2] = {1, 1};
  CUtensorMapSwizzle swz = panel_w == 64 ? CU_TENSOR_MAP_SWIZZLE_128B
                                         : (panel_w == 32 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B);
  CUtensorMap m;
  CUresult r = fn(&m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, (void*)base, dims, strides, box, es,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, swz, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return false;
  cache[key] = m;
  *out = m;
  return true;
}

template <int RP, int EPI, bool SPLIT, int MODE, int SKIPM = 0>
nmd_status run(const Factor& fm, const Factor& fq, const TcParams& p, int grid, cudaStream_t s) {
  using C = Cfg<RP, SPLIT, MODE != 0, SKIPM != 0>;
  CUtensorMap th, tl, tl2;
  if (!tensor_map(fq.hi, fq.rows, RP, C::PANEL_W, C::BN, &th)) return NMD_ERR_CUDA;
  if (!tensor_map(fq.lo, fq.rows, RP, C::PANEL_W, C::BN, &tl)) return NMD_ERR_CUDA;
  if (!tensor_map(fq.lo2, fq.rows, RP, C::PANEL_W, C::BN, &tl2)) return NMD_ERR_CUDA;
  // W tiles: the M-side rows [0, m0 + M) of the M factor's bf16 copy, so
  // that the rows of a ragged last tile past the block read as zero
  CUtensorMap tw = th;
  if (C::WSMEM && !tensor_map(fm.hi, p.m0 + p.M, RP, C::PANEL_W, BM, &tw)) return NMD_ERR_CUDA;
  // the shared-memory attributes belong to the current device.  At r_pad <=
  // 64 the carveout asks for the largest shared-memory configuration (228 KB
  // per SM): with the 166 KB of a CTA an SM would otherwise be set to 196 KB,
  // leaving no room for an update block (37 KB) beside it, and the deferred
  // update would run only on the SMs the grid leaves free.  (At r_pad = 256
  // the same setting slowed the sweep by 15%: there nothing fits beside a
  // CTA, and the L1 it takes away is lost.)
  static std::atomic<int> attr_set[kMaxDevices];
  if (!per_device(attr_set, [] {
        return (cudaFuncSetAttribute(panel_tc_kernel<RP, EPI, SPLIT, MODE, SKIPM>,
                                     cudaFuncAttributeMaxDynamicSharedMemorySize, (int)C::SMEM) == cudaSuccess &&
                (RP > 64 || cudaFuncSetAttribute(panel_tc_kernel<RP, EPI, SPLIT, MODE, SKIPM>,
                                                 cudaFuncAttributePreferredSharedMemoryCarveout,
                                                 100) == cudaSuccess)) ? 1 : 0;
      }))
    return NMD_ERR_CUDA;
  const unsigned gz = p.ksplit ? (unsigned)((p.K + p.ksplit - 1) / p.ksplit) : 1u;
  panel_tc_kernel<RP, EPI, SPLIT, MODE, SKIPM><<<dim3((unsigned)grid, C::RHALF ? 2u : 1u, gz), kThreads, C::SMEM, s>>>(
      th, tl, tl2, tw, p);
  return NMD_OK;
}

template <int RP, int MODE>
nmd_status dispatch_rp(int epilogue, bool split, const Factor& fm, const Factor& fq, const TcParams& p, int grid,
                       cudaStream_t s) {
  if constexpr (MODE == 2) {
    return run<RP, 0, true, 2>(fm, fq, p, grid, s);   // nearest neighbours: always the split pieces
  } else if constexpr (MODE == 1) {
    return split ? run<RP, 0, true, 1>(fm, fq, p, grid, s) : run<RP, 0, false, 1>(fm, fq, p, grid, s);
  }
  if (epilogue == NMD_EPI_DELTA && p.rmask != nullptr) {
    if (split) return run<RP, 1, true, 0, 2>(fm, fq, p, grid, s);
    return run<RP, 1, false, 0, 2>(fm, fq, p, grid, s);
  }
  if (epilogue == NMD_EPI_DELTA && p.skip_on) {
    if (split) return run<RP, 1, true, 0, 1>(fm, fq, p, grid, s);
    return run<RP, 1, false, 0, 1>(fm, fq, p, grid, s);
  }
  if (split)
    return epilogue == NMD_EPI_DELTA ? run<RP, 1, true, 0>(fm, fq, p, grid, s)
                                     : run<RP, 0, true, 0>(fm, fq, p, grid, s);
  return epilogue == NMD_EPI_DELTA ? run<RP, 1, false, 0>(fm, fq, p, grid, s)
                                   : run<RP, 0, false, 0>(fm, fq, p, grid, s);
}

template <int MODE>
nmd_status dispatch(int rp, int epilogue, bool split, const Factor& fm, const Factor& fq, const TcParams& p,
                    int grid, cudaStream_t s) {
  switch (rp) {
    case 16: return dispatch_rp<16, MODE>(epilogue, split, fm, fq, p, grid, s);
    case 32: return dispatch_rp<32, MODE>(epilogue, split, fm, fq, p, grid, s);
    case 64: return dispatch_rp<64, MODE>(epilogue, split, fm, fq, p, grid, s);
    case 128: return dispatch_rp<128, MODE>(epilogue, split, fm, fq, p, grid, s);
    case 256: return dispatch_rp<256, MODE>(epilogue, split, fm, fq, p, grid, s);
  }
  return NMD_ERR_UNSUPPORTED;
}

}  // namespace

// (of the chunk-skipping kernels)
int panel_chunk_rows(int rp, int precision) {
  const bool split = precision == NMD_FP32;
  switch (rp) {
    case 16: return split ? Cfg<16, true, false, true>::BN : Cfg<16, false, false, true>::BN;
    case 32: return split ? Cfg<32, true, false, true>::BN : Cfg<32, false, false, true>::BN;
    case 64: return split ? Cfg<64, true, false, true>::BN : Cfg<64, false, false, true>::BN;
    case 128: return split ? Cfg<128, true, false, true>::BN : Cfg<128, false, false, true>::BN;
    default: return split ? Cfg<256, true, false, true>::BN : Cfg<256, false, false, true>::BN;
  }
}

bool tc_supported(int rp, int precision) {
  if (precision == NMD_SIMT) return false;
  return rp == 16 || rp == 32 || rp == 64 || rp == 128 || rp == 256;
}

// R = sum over the splits of the partial R's, in split order
__global__ void split_reduce_kernel(const float* __restrict__ part, int64_t stride, int splits,
                                    float* __restrict__ R, int64_t n) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    float v = part[i];
    for (int z = 1; z < splits; ++z) v += part[z * stride + i];
    R[i] = v;
  }
}

nmd_status launch_panel_tc(const StepArgs& a, float* R, int* status, int* counter, int num_sms, cudaStream_t s,
                           int64_t* launches, float* Lout, float* rpart, int64_t rpart_rows) {
  if (!tc_supported(a.rp, a.precision)) return NMD_ERR_UNSUPPORTED;
  TcParams p{a.m0, a.M, a.q0, a.K, a.fm->hi, a.fm->lo, R, nullptr, status, Lout, nullptr, nullptr,
             (unsigned long long*)counter, a.skip_zero ? 1 : 0, 0, 0, a.rmask, a.rwords};
  const int64_t ntiles = (a.M + BM - 1) / BM;
  // a step with fewer tiles than SMs (the exact steps: b rows against all of
  // the other factor) splits K so that tiles x splits fill the SMs, each split
  // keeping at least 8 chunks; the partial R's are summed in split order
  int64_t splits = 1;
  if (Lout == nullptr && rpart != nullptr && ntiles < num_sms) {
    splits = std::min<int64_t>({(int64_t)num_sms / ntiles, (a.K + 64 * 8 - 1) / (64 * 8), 16,
                                rpart_rows / (ntiles * BM)});
    if (splits < 2) splits = 1;
  }
  int grid;
  if (splits > 1) {
    p.ksplit = ((a.K + splits - 1) / splits + 127) / 128 * 128;   // whole chunks of 64 or 128 rows
    splits = (a.K + p.ksplit - 1) / p.ksplit;
    p.R = rpart;
    p.rstride = a.M * a.rp;
    grid = (int)ntiles;
  } else {
    // fewest CTAs that keep the same number of tile rounds: the SMs left over
    // run the side-stream kernels of the step
    const int64_t rounds = (ntiles + num_sms - 1) / num_sms;
    grid = (int)((ntiles + rounds - 1) / rounds);
  }
  nmd_status st = dispatch<0>(a.rp, a.epilogue, a.precision == NMD_FP32, *a.fm, *a.fq, p, grid, s);
  if (st != NMD_OK) return st;
  ++*launches;
  if (splits > 1) {
    const int64_t n = a.M * a.rp;
    const int64_t blocks = std::min<int64_t>((n + 255) / 256, (int64_t)num_sms * 8);
    split_reduce_kernel<<<(unsigned)blocks, 256, 0, s>>>(rpart, p.rstride, (int)splits, R, n);
    ++*launches;
  }
  return NMD_OK;
}

void launch_wait_selftest(int* status, uint64_t limit_ns, cudaStream_t s) {
  wait_selftest_kernel<<<1, 32, 0, s>>>(status, limit_ns);
}

nmd_status launch_update_tc(const StepArgs& a, const float* R, const float* Rs, const uint8_t* flags,
                            const Factor& gi, float eta, float gamma, bool momentum, int* status, cudaStream_t s) {
  if (a.M <= 0) return NMD_OK;
  TcParams p{0, a.M, 0, a.rp, nullptr, nullptr, nullptr, nullptr, status, nullptr, nullptr, nullptr, nullptr, 0,
             0, 0, nullptr, 0, nullptr, R, Rs, flags, a.fm->master, a.fm->E, a.fm->hi, a.m0, eta, gamma,
             momentum ? 1 : 0, a.epilogue == NMD_EPI_DELTA ? 1 : 0};
  // One tile per CTA: a deferred update shares the GPU with the next step's
  // dense kernel, on the SMs its grid leaves free, and CTAs that retire every
  // few microseconds let the next step's G^{-1} kernel (higher priority, 188 KB
  // of shared memory) have one of those SMs.  With persistent CTAs it waited
  // for the whole deferred update: 583 us for the Gram chain of a 69,627-row
  // step against 311 us of dense kernel.
  const int64_t ntiles = (a.M + BM - 1) / BM;
  if (a.rp != 256) return NMD_ERR_UNSUPPORTED;
  return run<256, 0, true, 3>(*a.fm, gi, p, (int)ntiles, s);
}

nmd_status launch_nearest_tc(const Factor& f, int64_t N, int rp, unsigned long long* keys, int* status,
                             int num_sms, cudaStream_t s) {
  if (!tc_supported(rp, NMD_FP32)) return NMD_ERR_UNSUPPORTED;
  TcParams p{0, N, 0, N, f.hi, f.lo, nullptr, nullptr, status, nullptr, nullptr, nullptr, nullptr, 0, 0, 0,
             nullptr, 0, keys};
  const int64_t ntiles = (N + BM - 1) / BM;
  const int64_t rounds = (ntiles + num_sms - 1) / num_sms;
  const int grid = (int)((ntiles + rounds - 1) / rounds);
  return dispatch<2>(rp, 0, true, f, f, p, grid, s);
}

nmd_status launch_loss_dense_tc(const nmd_handle* h, double* parts, int maxparts, int* nparts, int* status,
                                cudaStream_t s, int64_t* launches) {
  if (!tc_supported(h->rp, h->opt.precision)) return NMD_ERR_UNSUPPORTED;
  TcParams p{0, h->m, 0, h->n, h->W.hi, h->W.lo, nullptr, parts, status, nullptr, h->ws.rowptr, h->ws.col,
             nullptr, 0, 0, 0};
  int64_t ntiles = (h->m + BM - 1) / BM;
  int grid = (int)(ntiles < h->num_sms ? ntiles : h->num_sms);
  if (grid > maxparts) grid = maxparts;
  nmd_status st = dispatch<1>(h->rp, 0, h->opt.precision == NMD_FP32, h->W, h->B, p, grid, s);
  if (st == NMD_OK) {
    ++*launches;
    *nparts = grid;
  }
  return st;
}

}  // namespace nmd
