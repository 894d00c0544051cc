// Tensor-core Newton-Schulz chain for sm_103a: tcgen05.mma (bf16 operands,
// fp32 accumulators in TMEM) on CTA pairs (cta_group::2, one 256-row tile of
// 256 or 128 columns per pair), operands staged by TMA into 128-byte-swizzled
// shared memory; one persistent launch runs all phases of all iterations (large
// batches: one phase, lm_api.cu says why).
//
// Per NS iteration (Section 2, odd-polynomial Newton-Schulz), with the
// normalisation X / (||G_hat||_F + eps) folded into iteration 0.  A wide
// matrix (s x l, s <= l) iterates as
//   GRAM : A  = X X^T          K = l, only tiles on or above the diagonal
//   POLY : B  = b A + c A A    K = s, only tiles on or above the diagonal;
//                              the epilogue reads the A tile
//   APPLY: X' = a X + B X      K = s, all tiles; the epilogue reads the X tile
//                              unless a is folded into B's diagonal
// and a tall one (l x s, kept in its own orientation) as A = X^T X and
// X' = a X + X B, which is the same function (p(X X^T) X = X p(X^T X)).
// A and A A are symmetric, so A A = A A^T and X B = X B^T: every operand is
// either K-major rows or MN-major columns of a stored matrix.
//
// A cluster of two CTAs computes one tile: CTA r holds rows [128 r, 128 r +
// 128) of the A operand and half of the B operand's N-rows, the pair's MMA
// (issued by CTA 0) leaves rows 128 r .. of the tile in CTA r's TMEM.  Each SM
// thus stages and reads half of B, which halves the shared-memory traffic per
// FLOP of a one-CTA tile.
//
// What bounds it: with 256-column tiles and long queues the operand feed, 32 KB
// per CTA and 64-deep K block, 11.6 TB/s from L2 (430 ns a block against 270 ns
// of MMAs, d = 768 set); with few tiles the latency of a tile, about 0.5 us
// for the counter, 3.3 us of MMAs (K = 768, half of that on 128 columns), 1.3 us
// for the epilogue, 1.5 us until the stores are complete and counted.
// Measured on one box against one launch per phase with the epilogue warps
// storing and waiting: 124M-shaped Muon step 1720 -> 1518 us, small sets
// (2 layers, d = 128) 193 -> 109 us, one d = 768 layer from a graph 338 -> 231
// us, three-piece 4-layer d = 1280 set 8030 -> 7460 us.  Large batches, which are
// power-capped, take a launch per phase: that set 7300-7630 us over the GPUs
// measured, the 720M-shaped set 14.2-14.7 ms for a Muon and a Lion step, no
// different beyond noise from the kernel before the chain.
//
// CTA roles (384 threads, one CTA per SM; 12 warps, three per sub-partition):
//   warp 0    TMA producer (one lane), smem ring (TcLayout); both CTAs' copies
//             signal CTA 0's full barrier
//   warp 1    TMEM allocator (both CTAs) + MMA issuer (CTA 0, one lane)
//   warps 2-9 epilogue: tcgen05.ld from TMEM, fused polynomial combination,
//             results written into shared memory (over the aux tile).  Warps
//             2-5 (one per TMEM lane quadrant and SM sub-partition) cover the
//             whole tile; warps 6-9 work only where the main products are
//             summed in registers (kPromo, half the columns each) and in a
//             launch whose parameter write reads W from global memory
//             (latency-bound), and all eight sum the split-K parts.  Eight
//             epilogue warps elsewhere measured
//             1 to 4% slower per Muon step on the d = 768 and 1280 sets: two of
//             them share each sub-partition's issue slots with the producer or
//             the MMA issuer.
//   warp 10   mover: TMA of the tile the epilogue combines with the
//             accumulator (A, X or W) into the aux buffer, the result stores
//             from it, and the count of a tile once its stores are complete
//   warp 11   scout: waits for the tiles' dependencies ahead of the producer
// The last APPLY of a Muon step can also apply the parameter update
// W <- W - eta_M (s X_K + lambda W) (Algorithm 1, Muon branch) in its
// epilogue, and X_K itself is never stored.  Where a is folded into B' (the
// default), the mover brings the W tile by TMA, the epilogue updates it in
// shared memory from the accumulator and the mover stores it back (a W tensor
// map per matrix in global memory).  Otherwise the aux tile is X, X_K goes
// to shared memory as bf16, and each warp then reads its 32 rows of W with
// coalesced 16-byte loads, updates and writes them.
// Tiles are assigned to pairs on the host by a longest-first greedy balance
// of their K lengths (a contiguous range per pair and phase), or dealt out in
// snake order where the list is made on the device.
// Two accumulators in TMEM let the epilogue of one tile overlap the main loop
// of the next.  Every wait, on a barrier or a counter, is bounded in time; a
// wait that gives up sets LM_FLAG_TIMEOUT, makes the other roles (and, through
// the flag, the other pairs) stop, waits (bounded) for its own copies and MMAs,
// frees TMEM and returns.
#include <cuda_bf16.h>
#include <cudaTypedefs.h>

#include "lm_ns_tc_shared.cuh"

namespace lm {
namespace {

using namespace tc;    // PTX wrappers (lm_tc_ptx.cuh)
using namespace tcs;   // constants, stop check and end-of-launch handshake (lm_ns_tc_shared.cuh)

constexpr int kAccBufs = 2;                          // 256-column accumulators in TMEM
constexpr int kScoutWarp = kAuxWarp + 1;             // waits for the tiles' dependencies, ahead of the producer
// 12 warps: three per SM sub-partition, so 168 registers a thread (a 13th
// would halve a sub-partition's share to 128 and spill the epilogue)
constexpr int kChainThreads = 32 * (kScoutWarp + 1);
constexpr int kFuseBatch = 4;   // W loads in flight per thread in the global-memory parameter write
constexpr int kTmemCols = 512;
// Shared-memory layout per operand precision and tile width.
//   kP = 1 (bf16 operands), 256 columns: a 5-stage ring of 32 KB per CTA and
//     a 64 KB aux/staging buffer; 128 columns: 8 stages of 24 KB and 32 KB.
//   kP = 3 (fp32 operands held as three bf16 pieces hi + mid + lo, exact), 128
//     columns: a 3-stage ring of 72 KB per CTA (the epilogue reads its aux
//     values and writes its results through global memory).
template <int kP, int kBN>
struct TcLayout {
  static constexpr int kBBytes = kBN / 2 * BK * 2;        // a CTA's half of a B operand block
  static constexpr int kStages = kP == 3 ? 3 : (kBN == 256 ? 5 : 8);
  static constexpr int kStageBytes = kP * (kABytes + kBBytes);
  static constexpr int kBoxes = kBN / 64;
  static constexpr size_t kAuxOffset = (size_t)kStages * kStageBytes;
  static constexpr size_t kBarOffset = kAuxOffset + (kP == 1 ? kBoxes * kAuxBoxBytes : 0);
  static constexpr size_t kSmemBytes = 1024 /*align slack*/ + kBarOffset + 512;
  static_assert(kSmemBytes <= 232448, "shared memory of one CTA");
};

// Operands of one tile.  Wide groups hold X as s x l, tall groups as l x s
// (the parameter's own orientation):
//   GRAM  wide: A = X X^T, both operands K-major rows of X (K = l)
//         tall: A = X^T X, both operands MN-major columns of X (K = l)
//   POLY      : B = b A + c A A, operands rows of A (K = s)
//   APPLY wide: X' = a X + B X, rows of B and MN-major X (K = s)
//         tall: X' = a X + X B, K-major rows of X and rows of B (K = s)
// A and B are symmetric and only their 256 x 256 tiles on or above the
// diagonal are stored.  A row block r of A (or B) therefore reads K blocks
// k >= 256 r K-major from the stored tiles, and K blocks below 256 r as the
// transposed stored tile, i.e. MN-major.  The split falls on a 256 boundary,
// so both CTAs of a pair use the same layout for every K block.
struct OpSeg {
  int kb_end;                    // K blocks [previous end, kb_end)
  bool a_mn, b_mn;
  const CUtensorMap* map_a;
  const CUtensorMap* map_b;
};
// At most three ranges of K blocks, [kb_start, s0.kb_end), [s0.kb_end,
// s1.kb_end), ...; an empty one is skipped.  Named rather than an array, which
// indexed at run time would live in local memory.
struct TilePlan {
  int kb_start;   // first K block (split Gram tiles start inside K)
  OpSeg s0, s1, s2;
};
template <int kBN>
__device__ __forceinline__ TilePlan tile_plan(int phase, const NsGroup& g, const TcGroupMaps& mp, int cur,
                                              const NsTile& t, bool from_a = false) {
  TilePlan P;
  P.kb_start = 0;
  if (phase == NS_GRAM) {
    const int kb_end = t.kb1 != 0 ? (int)t.kb1 : g.l_pad / BK;
    P.kb_start = t.kb1 != 0 ? (int)t.kb0 : 0;
    const bool mn = g.tall != 0;
    P.s0 = P.s1 = P.s2 = OpSeg{kb_end, mn, mn, mn ? &mp.xmn[cur] : &mp.xk[cur], mn ? &mp.nxmn[cur] : &mp.nxk[cur]};
    return P;
  }
  const int nk = g.s_pad / BK;
  const int ka = min(t.tm * (BM / BK), nk);   // first K block on or above row block tm
  const int kn = min(t.tn * kBN / BM * (BM / BK), nk);   // the same for column block tn
  if (phase == NS_POLY) {            // A-operand rows tm, B-operand rows tn (tn >= tm)
    P.s0 = OpSeg{ka, true, true, &mp.amn, &mp.namn};
    P.s1 = OpSeg{kn, false, true, &mp.a, &mp.namn};
    P.s2 = OpSeg{nk, false, false, &mp.a, &mp.na};
    return P;
  }
  // APPLY: one operand is B, or A where B = b A was not formed (the same
  // upper-tile storage)
  if (!g.tall) {                     // rows tm of B, X MN-major
    P.s0 = OpSeg{ka, true, true, from_a ? &mp.amn : &mp.bmn, &mp.nxmn[cur]};
    P.s1 = P.s2 = OpSeg{nk, false, true, from_a ? &mp.a : &mp.b, &mp.nxmn[cur]};
  } else {                           // rows of X K-major, rows tn of B
    P.s0 = OpSeg{kn, false, true, &mp.xk[cur], from_a ? &mp.namn : &mp.nbmn};
    P.s1 = P.s2 = OpSeg{nk, false, false, &mp.xk[cur], from_a ? &mp.na : &mp.nb};
  }
  return P;
}


// Producer k-loop of one tile, specialised on the operand layouts (a loop
// with per-block layout branches measured ~12% slower end to end).
// K-major operand half: one 64 (K) x 128 box; MN-major: one 4-D box that
// fills both 64 (MN) x 64 (K) swizzle atoms (one copy instead of two
// measured ~2% faster).  Returns false if a wait gave up.
template <int kS>
struct ProducerRing {
  int stage;
  uint32_t ph;
  int armed[kS];
};
// kP pieces per operand: piece q of matrix mat is matrix mat + q * pstride
// of the tensor map; a stage holds the kP A pieces, then the kP B pieces.
// same: both operands are the same rows of the same matrix (a diagonal Gram
// or polynomial tile), so only the A boxes are loaded and the MMA reads them
// as B too.
template <bool AMN, bool BMN, int kP, int kBN>
__device__ __forceinline__ bool produce_range(ProducerRing<TcLayout<kP, kBN>::kStages>& R,
                                              ProducerLog<TcLayout<kP, kBN>::kStages>& log, uint8_t* smem,
                                              uint64_t* full, uint64_t* empty, volatile int* abort_flag,
                                              uint64_t wait_ns, uint32_t rank, int kb0, int kb1,
                                              const CUtensorMap* map_a, const CUtensorMap* map_b, int row_a,
                                              int col_b, int mat, int pstride, bool same) {
  using L = TcLayout<kP, kBN>;
  const uint32_t own = same ? (uint32_t)(kP * kABytes) : (uint32_t)L::kStageBytes;   // this CTA's bytes
  for (int kb = kb0; kb < kb1; ++kb) {
    if (!mbar_wait(&empty[R.stage], R.ph ^ 1u, abort_flag, wait_ns)) return false;
    uint8_t* sa = smem + (size_t)R.stage * L::kStageBytes;
    uint8_t* sb = sa + kP * kABytes;
    const uint32_t fb = peer_addr(&full[R.stage], 0);
    if (rank == 0) {
      mbar_arrive_expect_tx(&full[R.stage], 2u * own);
      R.armed[R.stage] = (int)R.ph;
    }
    log.bytes[R.stage] = own;
    log.n += 1u;
    const int k0 = kb * BK;
#pragma unroll
    for (int q = 0; q < kP; ++q) {
      if (!AMN) tma_load_3d(sa + q * kABytes, map_a, fb, k0, row_a, mat + q * pstride);
      else tma_load_4d(sa + q * kABytes, map_a, fb, 0, k0, row_a >> 6, mat + q * pstride);
    }
#pragma unroll
    for (int q = 0; q < kP && !same; ++q) {
      if (!BMN) tma_load_3d(sb + q * L::kBBytes, map_b, fb, k0, col_b, mat + q * pstride);
      else tma_load_4d(sb + q * L::kBBytes, map_b, fb, 0, k0, col_b >> 6, mat + q * pstride);
    }
    if (++R.stage == L::kStages) {
      R.stage = 0;
      R.ph ^= 1u;
    }
  }
  return true;
}

// MMA issue for K blocks [kb0, kb1) of one tile with fixed operand layouts.
// kP = 3: with A = A0 + A1 + A2 and B = B0 + B1 + B2 (each piece 2^-8 of the
// previous in magnitude) the six products of order up to 2^-16 are summed,
// A0B0 + A0B1 + A1B0 + A0B2 + A2B0 + A1B1; the dropped ones are of order 2^-24.
// The tensor cores' fp32 accumulation loses about one unit of the last place of
// the accumulator per MMA, always in the same direction (2.2e-5 relative for a
// 1280-deep product with all six in one accumulator), so A0B0 has one of its
// own and the five smaller products, 2^-8 of it, share another (4.4e-6).
// kPromo (the full-fp32 mode): A0B0 is accumulated for one K block only (four
// MMAs), in one of two accumulators by turns, and the epilogue warps add each
// block's sum to theirs in fp32 registers, rounded to nearest, while the next
// block runs.  Five iterations of the quintic are then 0.2 to 0.63 times as far
// from fp64 as with fp32 FMAs on the CUDA cores (256 to 5120 wide: 4.5e-7 to
// 1.4e-6 against 1.6e-6 to 3.3e-6; dropping no product at all, eight of them,
// changes nothing).  Its cost: the warps that hold the sums cannot go on adding
// while they write a tile out, so the MMAs of the next tile wait (4-layer d =
// 1280 set: 10.7 ms per Muon step against 7.4-7.6 without).
// Main products: per K block n, accumulator n & 1; mfull: the block's four MMAs
// are done (both CTAs), mempty: every epilogue warp has read it.
struct MainRing {
  uint32_t n;          // K blocks issued
  uint32_t tmem;       // columns of accumulator 0
  uint64_t* mfull;
  uint64_t* mempty;
};
template <bool AMN, bool BMN, int kP, int kBN, bool kPromo>
__device__ __forceinline__ bool mma_range(int& stage, uint32_t& ph, uint8_t* smem, uint64_t* full,
                                          uint64_t* empty, volatile int* abort_flag, uint64_t wait_ns, int kb0,
                                          int kb1, uint32_t d_tmem, MainRing& mr, int kb_first, bool same) {
  using L = TcLayout<kP, kBN>;
  constexpr int qa[6] = {0, 0, 1, 0, 2, 1};
  constexpr int qb[6] = {0, 1, 0, 2, 0, 1};
  const uint32_t idesc = make_idesc(BM, kBN, AMN, BMN);
  for (int kb = kb0; kb < kb1; ++kb) {
    if (!mbar_wait(&full[stage], ph, abort_flag, wait_ns)) return false;
    tc_fence_after();
    const uint32_t sa = smem_u32(smem + (size_t)stage * L::kStageBytes);
    const uint32_t sb = same ? sa : sa + kP * kABytes;
    // descriptors of the stage's K = 0 slices; a 16-deep K step adds its
    // byte offset / 16 to the start-address field (bits 0-13: no carry, the
    // shared-memory window is below 2^18 bytes)
    const uint64_t a0 = AMN ? sw128_desc(sa, 64 * BK * 2, 1024) : sw128_desc(sa, 16, 1024);
    const uint64_t b0 = BMN ? sw128_desc(sb, 64 * BK * 2, 1024) : sw128_desc(sb, 16, 1024);
    auto step = [&](int m, int kk, uint32_t d, bool first) {
      const uint64_t adesc = a0 + (uint64_t)((qa[m] * kABytes + kk * (AMN ? 2048 : 32)) >> 4);
      const uint64_t bdesc = b0 + (uint64_t)((qb[m] * L::kBBytes + kk * (BMN ? 2048 : 32)) >> 4);
      umma_bf16(d, adesc, bdesc, idesc, first ? 0u : 1u);
    };
    if constexpr (kP == 1) {
#pragma unroll
      for (int kk = 0; kk < BK / 16; ++kk) step(0, kk, d_tmem, kb == kb_first && kk == 0);
    } else if constexpr (!kPromo) {
#pragma unroll
      for (int kk = 0; kk < BK / 16; ++kk)
#pragma unroll
        for (int m = 0; m < 6; ++m)
          step(m, kk, m == 0 ? d_tmem : d_tmem + (uint32_t)kBN, kb == kb_first && kk == 0 && m <= 1);
    } else {
      const uint32_t mb = mr.n & 1u;
      if (!mbar_wait(&mr.mempty[mb], ((mr.n >> 1) & 1u) ^ 1u, abort_flag, wait_ns)) return false;
      tc_fence_after();
#pragma unroll
      for (int kk = 0; kk < BK / 16; ++kk) step(0, kk, mr.tmem + mb * (uint32_t)kBN, kk == 0);
      umma_commit_pair(&mr.mfull[mb]);
      ++mr.n;
#pragma unroll
      for (int kk = 0; kk < BK / 16; ++kk)
#pragma unroll
        for (int m = 1; m < 6; ++m) step(m, kk, d_tmem, kb == kb_first && kk == 0 && m == 1);
    }
    umma_commit_pair(&empty[stage]);
    if (++stage == L::kStages) {
      stage = 0;
      ph ^= 1u;
    }
  }
  return true;
}

// fp32 value v as hi + mid + lo bf16 pieces, exactly: each piece takes the
// next 8 significant bits (the differences are exact in fp32).
__device__ __forceinline__ void split3(float v, float& h, float& m, float& l) {
  h = __bfloat162float(__float2bfloat16_rn(v));
  const float r1 = v - h;
  m = __bfloat162float(__float2bfloat16_rn(r1));
  l = r1 - m;
}
// The same for a pair of values, packed: the conversion to bf16 packs, and the
// halves are what is subtracted.
__device__ __forceinline__ void split3_pair(float a, float b, uint32_t& h, uint32_t& m, uint32_t& l) {
  h = pack_bf2(a, b);
  const float ra = a - bf_lo(h), rb = b - bf_hi(h);
  m = pack_bf2(ra, rb);
  l = pack_bf2(ra - bf_lo(m), rb - bf_hi(m));
}
// Epilogue of one 32 x 16 chunk (rows r0 .. r0 + 31, one per lane; columns
// j0 ..) with three-piece operands; aux values and results go through global
// memory in whole 32-byte sectors: lanes 2m and 2m + 1 access the two halves of
// row 2m, then of row 2m + 1, and exchange the halves that are not theirs.
//   kacc: APPLY's factor on the accumulator (1, or b where B = b A was not
//   formed).
//   aux: the A (POLY) or X (APPLY) element, hi + mid + lo; out: the result's
//   pieces, or fp32 in out_f32 (last APPLY).  base: element (r0, j0) of the
//   matrix in plane 0; ld: row length; plane: elements per piece.
struct AuxPieces {
  uint4 v[2][3];   // this lane's halves of rows 2m and 2m + 1, per plane
};
__device__ __forceinline__ void aux_load(AuxPieces& a, const __nv_bfloat16* aux, size_t plane, size_t base, size_t ld,
                                         int lane) {
  const size_t off0 = base + (size_t)(lane & ~1) * ld + ((lane & 1) ? 8 : 0);
#pragma unroll
  for (int k = 0; k < 2; ++k)
#pragma unroll
    for (int q = 0; q < 3; ++q)   // through L2: another SM may have written the tile in this launch
      a.v[k][q] = __ldcg(reinterpret_cast<const uint4*>(aux + q * plane + off0 + (size_t)k * ld));
}
// kAhead: a holds the chunk's aux values (not GRAM) and next, if next_ok, is the
// base of the chunk after it, whose aux values are loaded into a while this one
// is combined; without (register sums: no registers to spare) they are loaded
// here.
template <bool kAhead, typename Co>
__device__ __forceinline__ void piece_chunk(const float (&acc)[16], int phase, const Co& co, float nscale,
                                            float kacc, AuxPieces& a,
                                            const __nv_bfloat16* aux, __nv_bfloat16* out, float* out_f32,
                                            size_t plane, size_t base, size_t ld, bool row_ok, int j0, int ncols,
                                            bool next_ok, size_t next, int lane) {
  const bool odd = lane & 1;
  const size_t off0 = base + (size_t)(lane & ~1) * ld + (odd ? 8 : 0);   // this lane's half of row 2m
  float v[16];
  if (phase != NS_GRAM) {
    float h[2][8];   // this lane's halves of rows 2m and 2m + 1
#pragma unroll
    for (int k = 0; k < 2; ++k)
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        const uint4 a4 = kAhead ? a.v[k][q]
                                : __ldcg(reinterpret_cast<const uint4*>(aux + q * plane + off0 + (size_t)k * ld));
        const uint32_t aw[4] = {a4.x, a4.y, a4.z, a4.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          h[k][2 * e] = q == 0 ? bf_lo(aw[e]) : h[k][2 * e] + bf_lo(aw[e]);
          h[k][2 * e + 1] = q == 0 ? bf_hi(aw[e]) : h[k][2 * e + 1] + bf_hi(aw[e]);
        }
      }
    if (kAhead && next_ok) aux_load(a, aux, plane, next, ld, lane);
#pragma unroll
    for (int t = 0; t < 8; ++t) {   // an even lane owns row 2m, an odd one row 2m + 1
      const float got = __shfl_xor_sync(0xffffffffu, odd ? h[0][t] : h[1][t], 1);
      v[t] = odd ? got : h[0][t];
      v[8 + t] = odd ? h[1][t] : got;
    }
  }
  float o[16];
#pragma unroll
  for (int e = 0; e < 16; ++e) {
    if (phase == NS_GRAM) o[e] = acc[e] * nscale;
    else if (phase == NS_POLY) o[e] = poly_value(co.b, v[e], co.c, acc[e]);
    else o[e] = __fmaf_rn(co.a, v[e], kacc * acc[e]) * nscale;   // kacc = 1: exactly a v + acc, one rounding
    o[e] = (row_ok && j0 + e < ncols) ? o[e] : 0.f;
  }
  float h[2][8];
#pragma unroll
  for (int t = 0; t < 8; ++t) {
    const float got = __shfl_xor_sync(0xffffffffu, odd ? o[t] : o[8 + t], 1);
    h[0][t] = odd ? got : o[t];
    h[1][t] = odd ? o[8 + t] : got;
  }
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const size_t off = off0 + (size_t)k * ld;
    if (out_f32 != nullptr) {
      float4* dst = reinterpret_cast<float4*>(out_f32 + off);
      dst[0] = make_float4(h[k][0], h[k][1], h[k][2], h[k][3]);
      dst[1] = make_float4(h[k][4], h[k][5], h[k][6], h[k][7]);
      continue;
    }
    uint32_t w[3][4];
#pragma unroll
    for (int e = 0; e < 4; ++e) split3_pair(h[k][2 * e], h[k][2 * e + 1], w[0][e], w[1][e], w[2][e]);
#pragma unroll
    for (int q = 0; q < 3; ++q)
      *reinterpret_cast<uint4*>(out + q * plane + off) = make_uint4(w[q][0], w[q][1], w[q][2], w[q][3]);
  }
}

// ------------------------------- the chain ----------------------------------
// One launch runs a range of the (iteration, phase) sequence of every matrix
// of a batch.  Each pair walks its tiles of GRAM, POLY, APPLY, GRAM, ... in
// that order; what a tile reads is complete when the counters of its matrix
// say so (done: three counters per matrix, one per phase, each counting the
// epilogue warps that have stored their part of a tile), so a pair goes on to
// the next phase while other pairs finish the last one, and a whole
// iteration costs no launch, no TMEM or barrier set-up and no drain between
// phases.  A separate launch per phase measured 8 to 15 us whatever its work
// (bf16 msign of 768 x 3072: 320 us for 16 such launches).
//
// Every wait is for an item earlier in the sequence (iteration, GRAM < FINISH
// < POLY < APPLY) and every role works in that order, so with all pairs
// resident (a cooperative launch) none waits for ever.
struct ChainIter {
  float a, b, c;
  uint32_t mode;   // kIterFromA, kIterFold, and POLY phases run up to and including this iteration << 8
};
constexpr uint32_t kIterFromA = 1u;   // c = 0: B = b A is not formed, APPLY reads A and scales by b
constexpr uint32_t kIterFold = 2u;    // POLY adds a to B's diagonal (B' = a I + B), APPLY is X' = B' X
struct ChainParams {
  TcGroupMaps maps[kMaxGroupsTc];
  NsGroup groups[kMaxGroupsTc];
  const NsTile* tiles[3];
  const int* offsets[3];     // tiles of pair k: [offsets[k], offsets[k + 1]); NULL: dealt out in snake order
  int ntiles[3];             // (used without offsets)
  const int* counts;         // without offsets: device tile counts per phase, or NULL for ntiles
  const NsSplitTarget* targets;   // split Gram tiles
  const uint16_t* part_target;    // target of each part
  int ntargets;
  float* split_ws;
  uint32_t* parts_done;      // per target: epilogue warps that have written their share of a part
  uint32_t* done;            // 3 per matrix
  const double* norm2;
  float eps;
  int q0, q1;                // phases 3 * iteration + phase of this launch
  int steps;
  int nepi;                  // active epilogue warps per CTA: 4 or 8
  uint32_t sig;              // counts per tile: 1 per CTA (bf16) or 1 per epilogue warp (three pieces)
  uint32_t part_sig;         // counts per split-K part: 1 per epilogue warp
  // A split target is finished in fin_units units of 256 / fin_units rows,
  // each summed by one epilogue warp and counted once.
  int fin_units;
  unsigned* flags;
  FuseFinal fuse;            // fuse.mats != NULL: the last APPLY writes the parameters
  const unsigned char* active;
  uint64_t wait_ns;
  ChainIter it[kMaxNsSteps];
};

// The tiles of one pair in the order of the sequence, the next one always
// loaded ahead (its latency falls inside the current tile).
struct TileStream {
  int lo0, lo1, lo2, hi0, hi1, hi2;   // this pair's tiles per phase
  int pair, npairs;                   // npairs > 0: snake order over the list
  int it, ph, j, jend;
  int nit, nph;                       // the next tile's iteration and phase
  NsTile t;                           // the next tile
  bool have;
  __device__ __forceinline__ void fetch(const ChainParams& p) {
    for (;;) {
      if (j < jend) {
        const int k = npairs > 0 ? j * npairs + ((j & 1) ? npairs - 1 - pair : pair) : j;
        t = p.tiles[ph][k];
        nit = it;
        nph = ph;
        ++j;
        return;
      }
      if (++ph == 3) {
        ph = 0;
        ++it;
      }
      if (3 * it + ph >= p.q1) {
        have = false;
        return;
      }
      if (ph == NS_POLY && (p.it[it].mode & kIterFromA)) continue;
      j = ph == 0 ? lo0 : (ph == 1 ? lo1 : lo2);
      jend = ph == 0 ? hi0 : (ph == 1 ? hi1 : hi2);
    }
  }
};
__device__ __forceinline__ void pair_range(const ChainParams& p, int ph, int pair, int npairs, int& lo, int& hi) {
  if (p.offsets[ph] != nullptr) {
    lo = p.offsets[ph][pair];
    hi = p.offsets[ph][pair + 1];
    return;
  }
  // snake order: row r of npairs tiles is dealt left to right, then right to left
  const int n = p.counts != nullptr ? p.counts[ph] : p.ntiles[ph];
  const int full = n / npairs, rest = n - full * npairs;
  lo = 0;
  hi = full + (((full & 1) ? npairs - 1 - pair : pair) < rest ? 1 : 0);
}
__device__ __forceinline__ TileStream tile_stream(const ChainParams& p, int pair, int npairs) {
  TileStream S;
  pair_range(p, NS_GRAM, pair, npairs, S.lo0, S.hi0);
  pair_range(p, NS_POLY, pair, npairs, S.lo1, S.hi1);
  pair_range(p, NS_APPLY, pair, npairs, S.lo2, S.hi2);
  S.pair = pair;
  S.npairs = p.offsets[NS_GRAM] != nullptr ? 0 : npairs;
  S.it = p.q0 / 3;
  S.ph = p.q0 % 3 - 1;
  S.j = S.jend = 0;
  S.have = true;
  S.t = NsTile{};
  S.fetch(p);
  return S;
}

// What a tile reads: GRAM the X of the last APPLY, POLY the A, APPLY the B (or
// A where B is not formed; its X is complete when that A is).
__device__ __forceinline__ bool tile_ready(const ChainParams& p, int ph, int it, const NsGroup& g, int mat,
                                           volatile int* abort_flag) {
  const uint32_t* c = p.done + 3 * (size_t)(g.first_mat + mat);
  uint32_t need;
  if (ph == NS_GRAM) {
    if (it == 0) return true;
    c += NS_APPLY;
    need = (uint32_t)it * (uint32_t)g.n_apply * p.sig;
  } else if (ph == NS_POLY || (p.it[it].mode & kIterFromA)) {
    need = (uint32_t)(it + 1) * ((uint32_t)g.n_gram * p.sig + (uint32_t)(g.n_split * p.fin_units));
  } else {
    c += NS_POLY;
    need = (p.it[it].mode >> 8) * (uint32_t)g.n_poly * p.sig;
  }
  return counter_wait(c, need, p.flags, abort_flag, p.wait_ns);
}

// Rows [row0, row0 + nrows) of a split Gram target: the fp32 parts (already
// scaled), added in part order, as bf16 (or three bf16 planes) into A.  One
// warp, 8 columns a lane, two rows and four parts (16 loads) in flight.
template <int kBN>
__device__ __forceinline__ void finish_unit(const NsSplitTarget& T, const float* ws, int row0, int nrows, int lane) {
  constexpr int kPass = kBN == 256 ? 2 : 4;   // rows per trip, two of them per lane
  const int c = lane * 8 % kBN, rl = lane * 8 / kBN;
  if (c >= T.nc) return;
  __nv_bfloat16* dst = static_cast<__nv_bfloat16*>(T.a_tile);
  const int rend = min(row0 + nrows, T.nr);
  for (int r0 = row0; r0 < rend; r0 += kPass) {   // units start at multiples of 4 rows, T.nr is a multiple of 128
    const int r = r0 + rl * 2;
    const float* part = ws + (size_t)T.first * (BM * kBN) + (size_t)r * kBN + c;
    float v[2][8];
#pragma unroll
    for (int e = 0; e < 8; ++e) v[0][e] = v[1][e] = 0.f;
#pragma unroll 4
    for (int k = 0; k < T.nparts; ++k) {
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const float4* src = reinterpret_cast<const float4*>(part + (size_t)k * (BM * kBN) + u * kBN);
        const float4 x = __ldcg(src), y = __ldcg(src + 1);
        v[u][0] += x.x; v[u][1] += x.y; v[u][2] += x.z; v[u][3] += x.w;
        v[u][4] += y.x; v[u][5] += y.y; v[u][6] += y.z; v[u][7] += y.w;
      }
    }
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const size_t o = (size_t)(r + u) * T.ld + c;
      if (T.plane == 0) {
        *reinterpret_cast<uint4*>(dst + o) = make_uint4(pack_bf2(v[u][0], v[u][1]), pack_bf2(v[u][2], v[u][3]),
                                                        pack_bf2(v[u][4], v[u][5]), pack_bf2(v[u][6], v[u][7]));
        continue;
      }
      uint32_t w[3][4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        float h0, m0, l0, h1, m1, l1;
        split3(v[u][2 * e], h0, m0, l0);
        split3(v[u][2 * e + 1], h1, m1, l1);
        w[0][e] = pack_bf2(h0, h1);
        w[1][e] = pack_bf2(m0, m1);
        w[2][e] = pack_bf2(l0, l1);
      }
#pragma unroll
      for (int q = 0; q < 3; ++q)
        *reinterpret_cast<uint4*>(dst + q * T.plane + o) = make_uint4(w[q][0], w[q][1], w[q][2], w[q][3]);
    }
  }
}

__device__ __forceinline__ float as_float(uint32_t v) { return __uint_as_float(v); }
__device__ __forceinline__ float as_float(float v) { return v; }
// kN columns of a partial Gram product to its fp32 workspace row (zeros
// outside the true extent), in 32-byte stores.
template <typename V, int kN>
__device__ __forceinline__ void split_chunk(const V (&r)[kN], float* dst, float nscale, bool row_ok, int ncols) {
#pragma unroll
  for (int e = 0; e < kN; e += 8) {
    float o[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) o[u] = (row_ok && e + u < ncols) ? as_float(r[e + u]) * nscale : 0.f;
    st_global_v8(dst + e, o);
  }
}

// ----------------------------- bf16 epilogue --------------------------------
// What the epilogue does with an accumulator is fixed over a tile, so each
// form has a loop of its own that fits the instruction cache of an SM
// sub-partition.  One loop with the forms as (uniform) branches inside took 700
// cycles per 32-column chunk, most of them waiting for instructions, 5 to 8 us
// per tile against 3.3 us of MMAs at K = 768: the epilogue set the length of
// every phase of the d = 768 sets.
enum EpiForm {
  kEpiPlain,      // the accumulator (APPLY X' = B' X; GRAM)
  kEpiScale,      // ... times the normalisation of iteration 0
  kEpiPoly,       // b A + c acc, with k2 added on the diagonal (B' = a I + B)
  kEpiAxpy,       // (a X + k acc) * scale: APPLY without the fold
  kEpiW           // the parameter write on the W tile
};
struct EpiArgs {
  float k0, k1, k2, k3;   // Scale: k0; Poly: b, c, a; Axpy: a, k, scale; W: scale, s, eta_M, lambda
  int i, nrows, ncols;    // this lane's row, true extents (padding outside them is stored as zero)
  int diag;               // Poly: first column of the chunk that holds this warp's diagonal, -1: none
};
// One 32-column chunk, columns j0 .., accumulator row in r: 16-byte chunk c of
// row `row` of a box sits at chunk position c ^ (row mod 8).
template <int kForm, bool kMask>
__device__ __forceinline__ void epi_chunk(const uint32_t (&r)[32], uint8_t* box_row, int c0, int rx, int j0,
                                          const EpiArgs& a) {
  constexpr bool kAux = kForm != kEpiPlain && kForm != kEpiScale;
  uint4 x[4];   // all aux values before the first store (which may alias them as far as the compiler knows)
  if constexpr (kAux) {
#pragma unroll
    for (int u = 0; u < 4; ++u) x[u] = *reinterpret_cast<const uint4*>(box_row + (((c0 + u) ^ rx) << 4));
  }
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    uint4* cell = reinterpret_cast<uint4*>(box_row + (((c0 + u) ^ rx) << 4));
    float v[8];
    if constexpr (kAux) {
      const uint32_t xw[4] = {x[u].x, x[u].y, x[u].z, x[u].w};
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        v[2 * e] = bf_lo(xw[e]);
        v[2 * e + 1] = bf_hi(xw[e]);
      }
    }
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const float acc = __uint_as_float(r[u * 8 + e]);
      if constexpr (kForm == kEpiPlain) v[e] = acc;
      else if constexpr (kForm == kEpiScale) v[e] = acc * a.k0;
      else if constexpr (kForm == kEpiPoly) {
        if (e & 1) {   // pairs, in packed fp32: the same roundings as poly_value, half the instructions
          const float2 av = make_float2(__uint_as_float(r[u * 8 + e - 1]), acc);
          const float2 w = __ffma2_rn(make_float2(a.k0, a.k0), make_float2(v[e - 1], v[e]),
                                      __fmul2_rn(make_float2(a.k1, a.k1), av));
          v[e - 1] = w.x;
          v[e] = w.y;
        }
      } else if constexpr (kForm == kEpiAxpy) {
        v[e] = __fmaf_rn(a.k0, v[e], a.k1 * acc) * a.k2;   // the same rounding as ns_wide_kernel
      } else {
        // W <- W - eta_M (s X_K + lambda W) (Algorithm 1, Muon branch), with
        // X_K rounded to bf16 as it would have been stored
        const float xk = __bfloat162float(__float2bfloat16_rn(acc * a.k0));
        v[e] = __fsub_rn(v[e], __fmul_rn(a.k2, __fadd_rn(__fmul_rn(a.k1, xk), __fmul_rn(a.k3, v[e]))));
      }
    }
    if constexpr (kForm == kEpiPoly)
      if (j0 == a.diag) {   // uniform; one chunk of a diagonal tile per warp
#pragma unroll
        for (int e = 0; e < 8; ++e)
          if (a.i == j0 + u * 8 + e) v[e] += a.k2;
      }
    if constexpr (kMask) {
#pragma unroll
      for (int e = 0; e < 8; ++e) v[e] = (a.i < a.nrows && j0 + u * 8 + e < a.ncols) ? v[e] : 0.f;
    }
    *cell = make_uint4(pack_bf2(v[0], v[1]), pack_bf2(v[2], v[3]), pack_bf2(v[4], v[5]), pack_bf2(v[6], v[7]));
  }
}
// Boxes [b0, b1) (64 columns each) of a warp's 32 rows; the TMEM read of a
// chunk is in flight while the chunk before it is combined.  box_full: NULL
// when the boxes are not stored by the mover.
template <int kForm, bool kMask>
__device__ __forceinline__ void epi_boxes(uint32_t acc, uint8_t* rowbase, int rx, int b0, int b1, int col0,
                                          const EpiArgs& a, uint64_t* box_full, int lane) {
  uint32_t ra[32], rb[32];
  __syncwarp();   // tcgen05.ld is warp-collective: reconverge first
  tmem_ld32_async(acc + (uint32_t)(b0 * 64), ra);
#pragma unroll 1
  for (int b = b0; b < b1; ++b) {
    uint8_t* box_row = rowbase + b * kAuxBoxBytes;
    tmem_ld_wait(ra);
    tmem_ld32_async(acc + (uint32_t)(b * 64 + 32), rb);
    epi_chunk<kForm, kMask>(ra, box_row, 0, rx, col0 + b * 64, a);
    tmem_ld_wait(rb);
    if (b + 1 < b1) tmem_ld32_async(acc + (uint32_t)(b * 64 + 64), ra);
    epi_chunk<kForm, kMask>(rb, box_row, 4, rx, col0 + b * 64 + 32, a);
    if (box_full != nullptr) fence_proxy_async_smem();
    __syncwarp();
    if (box_full != nullptr && lane == 0) mbar_arrive(&box_full[b]);
  }
}

// ------------------------------- the kernel ---------------------------------
// kSplit: the Gram tiles include split-K parts (the plain instantiation keeps
// the common path free of them).  kP: bf16 pieces per operand value (1: bf16
// operands; 3: fp32 operands as hi + mid + lo bf16 pieces, six products).
template <bool kSplit, int kP, int kBN, bool kPromo>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kChainThreads, 1)
    ns_tc_kernel(const __grid_constant__ ChainParams p) {
  using L = TcLayout<kP, kBN>;
  constexpr int kStages = L::kStages;
  // tiles in flight in TMEM: kP = 1 double-buffers two accumulators; kP = 3
  // gives one tile both (main and cross products)
  constexpr int kAccRing = kAccBufs;
  constexpr int kAccCols = kP == 3 && !kPromo ? 2 * kBN : kBN;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~uintptr_t(1023));
  uint8_t* auxbuf = smem + L::kAuxOffset;   // kP = 1: 4 x (128 rows x 64 cols) bf16, 128-byte swizzled
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + L::kBarOffset);
  uint64_t* empty = full + kStages;
  uint64_t* accfull = empty + kStages;
  uint64_t* accempty = accfull + 2;
  uint64_t* aux_full = accempty + 2;
  uint64_t* done = aux_full + 1;
  uint64_t* box_full = done + 1;    // per 64-column box of auxbuf: results written, ready to store
  uint64_t* box_free = box_full + 4;   // all four stored (read by the TMA): auxbuf may be rewritten
  uint64_t* mfull = box_free + 1;      // three pieces: main-product accumulators (MainRing)
  uint64_t* mempty = mfull + 2;
  ProducerLog<kStages>* log = reinterpret_cast<ProducerLog<kStages>*>(mempty + 2);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(log + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  uint32_t* stop_word = tmem_slot + 2;
  uint32_t* aux_left = tmem_slot + 3;   // epilogue warps that have left a tile (parameter write through global memory)
  uint32_t* ready = tmem_slot + 4;   // tiles whose operands are complete (scout)

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_rank();          // 0: MMA issuer of the pair
  const int pair = blockIdx.x >> 1, npairs = gridDim.x >> 1;
  const int nepi = p.nepi;
  // The last APPLY of a Muon step may also write the parameters.  Where a is
  // folded into B' its aux tile is the W tile, updated in shared memory and
  // stored back by TMA; otherwise the aux tile is X and W is read from global
  // memory after the tile (that phase then has a launch of its own, with
  // eight epilogue warps for the latency).
  const bool fuse = p.fuse.mats != nullptr;
  // Workspace tile of a split-K part.  Only the three-piece mode, whose cap cuts
  // every long Gram tile, needs numbers past 16 bits (with them the bf16 epilogue
  // spills more: ragged d = 300 set 231 us a Muon step against 228).
  auto part_of = [](const NsTile& t) { return kP == 3 && !kPromo ? tc_part(t) : (int)t.slot - 1; };
  // epilogue reads the A (POLY) or X (APPLY) tile; an APPLY whose B has a
  // folded into its diagonal needs no X tile
  auto needs_aux = [&](int ph, int it) {
    if (kP != 1 || ph == NS_GRAM) return false;
    return ph == NS_POLY || !(p.it[it].mode & kIterFold) || (fuse && it == p.steps - 1);
  };

  if (p.counts != nullptr) {
    // masked launch with nothing selected: every CTA leaves before any
    // barrier, TMEM or cluster work
    griddep_wait();
    if (p.counts[NS_GRAM] == 0) {
      griddep_launch_dependents();
      return;
    }
  }

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < kAccBufs; ++b) {
      mbar_init(&accfull[b], 1);
      mbar_init(&accempty[b], 2 * nepi);
    }
    mbar_init(aux_full, 1);
    mbar_init(done, 1);
    for (int b = 0; b < 4; ++b) mbar_init(&box_full[b], 4);   // four warps (lane quadrants) write a box
    mbar_init(box_free, 1);
    for (int b = 0; b < 2; ++b) {
      mbar_init(&mfull[b], 1);
      mbar_init(&mempty[b], 2 * nepi);
    }
    log->n = 0;
    *abort_flag = 0;
    *aux_left = 0u;
    *ready = 0u;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    tmem_alloc(tmem_slot, kTmemCols);
    tmem_relinquish();
  }
  const bool stopped = pair_start(p.flags, stop_word, rank);   // an earlier launch gave up: no tiles
  const uint32_t tmem_base = *tmem_slot;
  const uint64_t wait_ns = p.wait_ns;

  auto give_up = [&]() {
    *abort_flag = 1;
    atomicOr(p.flags, LM_FLAG_TIMEOUT);
  };

  ProducerRing<kStages> R;   // producer lane: ring position and armed phases
  R.stage = 0;
  R.ph = 0;
  for (int s = 0; s < kStages; ++s) R.armed[s] = -1;

  if (warp == 0) {
    // ------------------------------ producer ------------------------------
    if (lane == 0) {
      bool ok = true;
      uint32_t ntile = 0;
      for (TileStream S = tile_stream(p, pair, npairs); ok && !stopped && S.have;) {
        const NsTile t = S.t;
        const int it = S.nit, phase = S.nph;
        S.fetch(p);
        const NsGroup& g = p.groups[t.group];
        // a diagonal Gram or polynomial tile: the B rows are the A rows
        const bool same = kBN == BM && phase != NS_APPLY && t.tm == t.tn;
        const TilePlan P = tile_plan<kBN>(phase, g, p.maps[t.group], it & 1, t, (p.it[it].mode & kIterFromA) != 0u);
        if (!smem_counter_wait(ready, ++ntile, abort_flag, wait_ns)) {   // the scout has seen its operands
          give_up();
          break;
        }
        const int row_a = t.tm * BM + (int)rank * kHalf;
        const int col_b = t.tn * kBN + (int)rank * (kBN / 2);
        int kb0 = P.kb_start;
#pragma unroll 1
        for (int sg = 0; ok && sg < 3; ++sg) {
          const OpSeg S = sg == 0 ? P.s0 : (sg == 1 ? P.s1 : P.s2);
          if (S.kb_end <= kb0) continue;
          if (!S.a_mn && !S.b_mn)
            ok = produce_range<false, false, kP, kBN>(R, *log, smem, full, empty, abort_flag, wait_ns, rank, kb0, S.kb_end, S.map_a,
                                             S.map_b, row_a, col_b, t.mat, g.count,
                                             same);
          else if (!S.a_mn)
            ok = produce_range<false, true, kP, kBN>(R, *log, smem, full, empty, abort_flag, wait_ns, rank, kb0, S.kb_end, S.map_a,
                                            S.map_b, row_a, col_b, t.mat, g.count,
                                             same);
          else
            ok = produce_range<true, true, kP, kBN>(R, *log, smem, full, empty, abort_flag, wait_ns, rank, kb0, S.kb_end, S.map_a,
                                           S.map_b, row_a, col_b, t.mat, g.count,
                                             same);
          kb0 = S.kb_end;
        }
        if (!ok) give_up();
      }
    }
  } else if (warp == 1) {
    // ------------------------------ MMA issuer -----------------------------
    if (lane == 0 && rank == 0) {
      int stage = 0;
      uint32_t ph = 0;
      int ab = 0;
      uint32_t aph = 0;
      bool ok = true;
      MainRing mr{0u, tmem_base + (uint32_t)(2 * kBN), mfull, mempty};   // kP = 3: columns behind the cross products
      for (TileStream S = tile_stream(p, pair, npairs); ok && !stopped && S.have;) {
        const NsTile t = S.t;
        const int it = S.nit, phase = S.nph;
        S.fetch(p);
        const NsGroup& g = p.groups[t.group];
        // a diagonal Gram or polynomial tile: the B rows are the A rows
        const bool same = kBN == BM && phase != NS_APPLY && t.tm == t.tn;
        const TilePlan P = tile_plan<kBN>(phase, g, p.maps[t.group], it & 1, t, (p.it[it].mode & kIterFromA) != 0u);
        if (!mbar_wait(&accempty[ab], aph ^ 1u, abort_flag, wait_ns)) {
          give_up();
          break;
        }
        tc_fence_after();
        // three pieces: main and cross products, or with kPromo the cross
        // products alone
        const uint32_t d_tmem = tmem_base + (uint32_t)(ab * kAccCols);
        int kb0 = P.kb_start;
#pragma unroll 1
        for (int sg = 0; ok && sg < 3; ++sg) {
          const OpSeg S = sg == 0 ? P.s0 : (sg == 1 ? P.s1 : P.s2);
          if (S.kb_end <= kb0) continue;
          if (!S.a_mn && !S.b_mn)
            ok = mma_range<false, false, kP, kBN, kPromo>(stage, ph, smem, full, empty, abort_flag, wait_ns, kb0, S.kb_end, d_tmem, mr,
                                            P.kb_start, same);
          else if (!S.a_mn)
            ok = mma_range<false, true, kP, kBN, kPromo>(stage, ph, smem, full, empty, abort_flag, wait_ns, kb0, S.kb_end, d_tmem, mr,
                                            P.kb_start, same);
          else
            ok = mma_range<true, true, kP, kBN, kPromo>(stage, ph, smem, full, empty, abort_flag, wait_ns, kb0, S.kb_end, d_tmem, mr,
                                            P.kb_start, same);
          kb0 = S.kb_end;
        }
        if (!ok) give_up();
        if (!ok) break;
        umma_commit_pair(&accfull[ab]);
        if (++ab == kAccRing) {
          ab = 0;
          aph ^= 1u;
        }
      }
      // all issued MMAs complete before TMEM is released
      umma_commit_local(done);
      volatile int never = 0;
      mbar_wait(done, 0, &never, kCleanupWaitNs);
    }
  } else if (warp == kScoutWarp) {
    // -------------------------------- scout --------------------------------
    // Waits, tile by tile and as far ahead as the counters allow, until what a
    // tile reads is complete.  The operands were written by other SMs: the
    // counter acquires them, and the proxy fence orders them before the TMA
    // copies of this CTA that the release of `ready` lets start.  Polling in
    // the producer instead stalls its copies for the poll and the fence (about
    // 1 us) before every tile.
    if (lane == 0) {
      for (TileStream S = tile_stream(p, pair, npairs); !stopped && S.have;) {
        const NsTile t = S.t;
        const int it = S.nit, phase = S.nph;
        S.fetch(p);
        if (!tile_ready(p, phase, it, p.groups[t.group], t.mat, abort_flag)) {
          give_up();
          break;
        }
        fence_proxy_async();
        smem_counter_add(ready, 1u);
      }
    }
  } else if (warp == kAuxWarp) {
    // -------------------------------- mover --------------------------------
    // Everything between auxbuf and global memory, so that the epilogue warps
    // never wait for a copy.  Per tile: brings the aux tile (A for POLY, X for
    // an APPLY without the fold, W for a parameter write; W boxes past the
    // parameter's extent read zeros) while the tile's main loop runs, stores
    // each 64-column box of the results (128 rows of this CTA) as soon as the
    // epilogue warps have written it, gives the boxes back once the TMA has
    // read them and counts the tile once its stores are complete.
    if (lane == 0 && kP == 1) {
      uint32_t xph = 0, sph = 0, ntile = 0;
      int armed = -1;
      bool ok = true;
      for (TileStream S = tile_stream(p, pair, npairs); ok && !stopped && S.have;) {
        const NsTile t = S.t;
        const int it = S.nit, phase = S.nph;
        S.fetch(p);
        ++ntile;
        const NsGroup& g = p.groups[t.group];
        const TcGroupMaps& mp = p.maps[t.group];
        const bool fused = fuse && phase == NS_APPLY && it == p.steps - 1;
        const bool fold = (p.it[it].mode & kIterFold) != 0u;
        const int row0 = t.tm * BM + (int)rank * kHalf;
        const int m = g.first_mat + t.mat;
        if (needs_aux(phase, it)) {
          const CUtensorMap* map = (phase == NS_POLY) ? &mp.a : &mp.xk[it & 1];
          int zc = t.mat;
          if (fused && fold) {
            map = p.fuse.wmaps + m;
            zc = 0;
          } else {
            ok = smem_counter_wait(ready, ntile, abort_flag, wait_ns);   // A, or the X of this APPLY
          }
          // auxbuf is free: the stores of the tile before have read it (below);
          // a parameter write through global memory counts its tiles instead
          if (ok && fused && !fold)
            ok = smem_counter_wait(aux_left, (ntile - 1u) * (uint32_t)nepi, abort_flag, wait_ns);
          if (!ok) {
            give_up();
            break;
          }
          mbar_arrive_expect_tx(aux_full, L::kBoxes * kAuxBoxBytes);
          armed = (int)xph;
#pragma unroll
          for (int b = 0; b < L::kBoxes; ++b)
            tma_load_3d_local(auxbuf + b * kAuxBoxBytes, map, aux_full, t.tn * kBN + 64 * b, row0, zc);
          xph ^= 1u;
        }
        if ((kSplit && phase == NS_GRAM && t.slot != 0) || (fused && !fold)) continue;   // no TMA stores
        // the load maps (64 x 128 boxes) serve the stores too
        const CUtensorMap* dst = phase == NS_GRAM ? &mp.a : (phase == NS_POLY ? &mp.b : &mp.xk[(it & 1) ^ 1]);
        int zc = t.mat, nrow = phase == NS_APPLY && g.tall ? g.l_pad : g.s_pad;
        int ncol = phase == NS_APPLY && !g.tall ? g.l_pad : g.s_pad;
        if (fused) {   // boxes that reach into W
          dst = p.fuse.wmaps + m;
          zc = 0;
          nrow = (int)p.fuse.mats[m].rows;
          ncol = (int)p.fuse.mats[m].cols;
        }
#pragma unroll
        for (int b = 0; b < L::kBoxes; ++b) {
          if (ok) ok = mbar_wait(&box_full[b], sph, abort_flag, wait_ns);
          // a parameter write stops at a give-up that was recorded before it
          if (b == 0 && fused && (*reinterpret_cast<volatile unsigned*>(p.flags) & LM_FLAG_TIMEOUT) != 0u) nrow = 0;
          const int x0 = t.tn * kBN + 64 * b;
          if (ok && row0 < nrow && x0 < ncol) tma_store_3d(dst, auxbuf + b * kAuxBoxBytes, x0, row0, zc);
          bulk_commit();
        }
        if (!ok) {
          give_up();
          break;
        }
        sph ^= 1u;
        bulk_wait_read<0>();
        mbar_arrive(box_free);
        if (!fused) {
          bulk_wait_all();
          red_release_gpu(p.done + 3 * (size_t)m + phase, 1u);
        }
      }
      if (!ok && armed >= 0) {
        volatile int never = 0;
        mbar_wait(aux_full, (uint32_t)armed, &never, kCleanupWaitNs);
      }
      bulk_wait_all();
    }
  } else {
    // ------------------------------ epilogue -------------------------------
    // Thread (quadrant q, lane) owns one row of this CTA's half tile and half
    // (nepi = 8) or all (nepi = 4) of its columns, in 32-column chunks.
    // Results go into auxbuf (over the aux values, if any) in the 128-byte
    // swizzled box layout, and the mover sends each 64-column box on as
    // soon as it is written rather than all boxes at the end of the tile: all
    // pairs run tiles of equal length, so stores issued at tile end coincide
    // across the GPU and starve the operand loads (measured: 2846 -> 1568
    // cycles per APPLY tile of the MMA issuer waiting for operands).  The TMEM
    // read of a chunk is in flight while the chunk before it is combined.
    const int q = warp & 3;                   // TMEM lane quadrant of this warp
    const int half0 = nepi == 8 ? (warp - 2) >> 2 : 0;   // first half of the tile's columns it covers
    const int nhalves = 8 / nepi;
    const int row = q * 32 + lane;            // row of this CTA's half tile
    const uint32_t acc_empty0 = peer_addr(&accempty[0], 0);
    const uint32_t acc_empty1 = peer_addr(&accempty[kAccRing - 1], 0);
    const uint32_t mempty0 = peer_addr(&mempty[0], 0), mempty1 = peer_addr(&mempty[1], 0);
    int ab = 0;
    uint32_t aph = 0, xph = 0, sph = 0, ntile = 0;
    uint32_t nblk = 0;   // three pieces: K blocks whose main products this warp has added
    bool alive = !stopped;
    // Finish units of the split Gram tiles of one iteration, dealt out to all
    // eight warps of every CTA (loads in flight bound them); a warp reaches them
    // after its GRAM tiles and before its POLY tiles of that iteration.
    int fin_it = p.q0 / 3 + (p.q0 % 3 ? 1 : 0);
    const int fin_end = (p.q1 + 2) / 3;
    const int fin_first = (2 * pair + (int)rank) * kEpiWarps + warp - 2;
    int fin_u = fin_first;   // this warp's next unit of iteration fin_it
    int fin_seen = -1;       // last target whose parts are known to be complete
    // Runs this warp's units of iteration fin_it: all that are left (waiting
    // for their parts), or with `bar` only while their parts are complete and
    // the accumulator the warp will wait for is not (time it has to spare).
    auto finish = [&](const uint64_t* bar, uint32_t parity) {
      for (; fin_u < p.ntargets * p.fin_units; fin_u += 2 * npairs * kEpiWarps) {
        const int tg = fin_u / p.fin_units;
        const NsSplitTarget T = p.targets[tg];
        if (p.active != nullptr && !p.active[T.mat]) continue;
        if (bar != nullptr && __any_sync(0xffffffffu, mbar_try_wait_hint(const_cast<uint64_t*>(bar), parity, 1u))) return;
        if (tg != fin_seen) {
          const uint32_t* ctr = p.parts_done + tg;
          const uint32_t need = (uint32_t)(fin_it + 1) * (uint32_t)T.nparts * p.part_sig;
          if (bar != nullptr) {
            if (!__all_sync(0xffffffffu, (int32_t)(ld_acquire_gpu(ctr) - need) >= 0)) return;
          } else if (!__all_sync(0xffffffffu, counter_wait(ctr, need, p.flags, abort_flag, wait_ns))) {
            if (lane == 0) give_up();
            alive = false;
            return;
          }
          fin_seen = tg;
        }
        finish_unit<kBN>(T, p.split_ws, (fin_u % p.fin_units) * (BM / p.fin_units), BM / p.fin_units, lane);
        __syncwarp();
        if (lane == 0) red_release_gpu(p.done + 3 * (size_t)T.mat + NS_GRAM, 1u);
      }
      if (bar != nullptr) return;
      ++fin_it;
      fin_u = fin_first;
      fin_seen = -1;
    };
    TileStream S = tile_stream(p, pair, npairs);
    while (alive && S.have && warp - 2 < nepi) {
      const NsTile t = S.t;
      const int it = S.nit, phase = S.nph;
      S.fetch(p);
      ++ntile;
      const int cur = it & 1;
      if (kSplit) {
        while (alive && (fin_it < it || (fin_it == it && phase != NS_GRAM))) finish(nullptr, 0u);
        if (!alive) break;
        if (phase == NS_GRAM && fin_it == it)
          finish(!kPromo ? &accfull[ab] : &mfull[nblk & 1u], !kPromo ? aph : (nblk >> 1) & 1u);
      }
      const NsGroup& g = p.groups[t.group];
      const ChainIter co = p.it[it];
      const bool fold = (co.mode & kIterFold) != 0u;
      const bool aux_phase = needs_aux(phase, it);
      const bool fused = phase == NS_APPLY && fuse && it == p.steps - 1;
      const bool fuse_w_tile = kP == 1 && fused && fold;
      const MatDesc* fd = fused ? &p.fuse.mats[g.first_mat + t.mat] : nullptr;
      const bool global_w = kP == 1 && fused && !fold;
      // a tile whose epilogue starts after a give-up was recorded leaves W alone
      // (another matrix's non-finite norm, in the same word, does not stop it)
      const unsigned flags_now = global_w && lane == 0 ? *reinterpret_cast<volatile unsigned*>(p.flags) : 0u;
      const bool write_w = global_w && (__shfl_sync(0xffffffffu, flags_now, 0) & LM_FLAG_TIMEOUT) == 0u;
      bool ok = true;
      // three pieces: half the tile's columns per warp; the main products of
      // each K block, added in block order
      float sum[kPromo ? 2 : 1][kPromo ? 32 : 1];
      if constexpr (kPromo) {
        const int nk = phase != NS_GRAM ? g.s_pad / BK : (t.kb1 != 0 ? (int)t.kb1 - (int)t.kb0 : g.l_pad / BK);
        const uint32_t main0 = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(2 * kBN + half0 * (kBN / 2));
#pragma unroll
        for (int e = 0; e < 32; ++e) sum[0][e] = sum[1][e] = 0.f;
#pragma unroll 1
        for (int k = 0; ok && k < nk; ++k, ++nblk) {
          const uint32_t mb = nblk & 1u;
          ok = mbar_wait_warp(&mfull[mb], (nblk >> 1) & 1u, abort_flag, wait_ns);
          if (!ok) break;
          tc_fence_after();
          uint32_t ra[32], rb[32];
          tmem_ld32_async(main0 + mb * (uint32_t)kBN, ra);
          tmem_ld32_async(main0 + mb * (uint32_t)kBN + 32u, rb);
          tmem_ld_wait(ra);
          tmem_ld_wait(rb);
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive_cluster(mb == 0u ? mempty0 : mempty1);
#pragma unroll
          for (int e = 0; e < 32; ++e) {
            sum[0][e] += __uint_as_float(ra[e]);
            sum[1][e] += __uint_as_float(rb[e]);
          }
        }
      }
      if (ok) ok = mbar_wait_warp(&accfull[ab], aph, abort_flag, wait_ns);
      if (ok && aux_phase) ok = mbar_wait_warp(aux_full, xph, abort_flag, wait_ns);
      if (!ok) {
        if (lane == 0) give_up();
        alive = false;
        break;
      }
      tc_fence_after();
      // this epilogue reads its aux values with generic loads: acquire what
      // the scout has seen (this tile is in it: its MMAs are done)
      if (kP == 3 && phase != NS_GRAM) (void)smem_counter_read(ready);

      // APPLY: X' = a X + B X, or a X + b (A X) where B = b A was not formed
      const float kacc = (co.mode & kIterFromA) ? co.b : 1.f;
      float nscale = 1.f;
      if (it == 0) {
        const float n = (float)sqrt(p.norm2[g.first_mat + t.mat]) + p.eps;
        nscale = (phase == NS_GRAM) ? 1.f / (n * n) : (phase == NS_APPLY ? 1.f / n : 1.f);
      }
      // output extents: s x s (GRAM, POLY), s x l (APPLY wide), l x s (APPLY tall)
      const bool apply_tall = phase == NS_APPLY && g.tall;
      const int nrows = apply_tall ? g.l : g.s;
      const int row_lim = apply_tall ? g.l_pad : g.s_pad;
      const int ncols = (phase == NS_APPLY) ? (g.tall ? g.s : g.l) : g.s;
      const int jmax = (phase == NS_APPLY) ? (g.tall ? g.s_pad : g.l_pad) : g.s_pad;
      const int r0 = t.tm * BM + (int)rank * kHalf + q * 32;   // first row of this warp
      const int i = r0 + lane;
      const bool warp_in = r0 < row_lim;        // rows past the padded matrix are skipped
      const bool split = kSplit && phase == NS_GRAM && t.slot != 0;
      if (fused && lane == 0 && q == 0 && half0 == 0 && rank == 0 && t.tm == 0 && t.tn == 0 &&
          !isfinite((float)sqrt(p.norm2[g.first_mat + t.mat])))
        atomicOr(p.flags, LM_FLAG_NONFINITE);
      const uint32_t acc0 = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(ab * kAccCols);
      if constexpr (kP == 3) {
        // rows of the output: s_pad or l_pad (APPLY tall); ld its row length
        const size_t ld = (size_t)(phase == NS_APPLY ? (g.tall ? g.s_pad : g.l_pad) : g.s_pad);
        const size_t msize = (size_t)(phase == NS_APPLY ? (size_t)g.s_pad * g.l_pad : (size_t)g.s_pad * g.s_pad);
        const size_t plane = (size_t)g.count * msize;
        const __nv_bfloat16* aux = static_cast<const __nv_bfloat16*>(phase == NS_POLY ? g.A : g.X[cur]);
        __nv_bfloat16* out = static_cast<__nv_bfloat16*>(phase == NS_GRAM ? g.A : (phase == NS_POLY ? g.B : g.X[cur ^ 1]));
        float* out_f32 = (phase == NS_APPLY && it == p.steps - 1) ? static_cast<float*>(g.Xf) : nullptr;
        // One 16-column chunk, columns [c0, c0 + 16) of the tile, next c0 + 16
        // of this warp's columns up to c1.  A chunk's aux values are loaded one
        // chunk ahead, the first before the accumulators are read.
        const size_t tile0 = (size_t)t.mat * msize + (size_t)r0 * ld + (size_t)t.tn * kBN;
        const int first = kPromo ? half0 * (kBN / 2) : 0, c1 = kPromo ? first + kBN / 2 : kBN;
        auto inside = [&](int c0) { return warp_in && c0 < c1 && t.tn * kBN + c0 < jmax; };   // the padded matrix
        AuxPieces ap;
        if (!kPromo && phase != NS_GRAM && inside(first)) aux_load(ap, aux, plane, tile0 + first, ld, lane);
        auto emit = [&](const float (&x)[16], int c0) {
          const int j = t.tn * kBN + c0;
          if (!inside(c0)) return;
          if (split)
            split_chunk(x, p.split_ws + (size_t)part_of(t) * (BM * kBN) + (size_t)((int)rank * kHalf + row) * kBN + c0,
                        nscale, i < nrows, ncols - j);
          else
            piece_chunk<!kPromo>(x, phase, co, nscale, kacc, ap, aux, out, out_f32, plane, tile0 + c0, ld, i < nrows, j, ncols,
                        !kPromo && inside(c0 + 16), tile0 + c0 + 16, lane);
        };
        // Chunks go through one loop body (unrolled, the copies ran at the pace
        // of instruction fetch: 7 us per tile).
        if constexpr (kPromo) {   // half the columns: add the cross products, move the sums down between chunks
          const int cc = half0 * (kBN / 2);
#pragma unroll
          for (int c = 0; c < 2; ++c) {
            uint32_t rc[32];
            __syncwarp();   // tcgen05.ld is warp-collective: reconverge first
            tmem_ld32_async(acc0 + (uint32_t)(cc + c * 32), rc);
            tmem_ld_wait(rc);
#pragma unroll
            for (int e = 0; e < 32; ++e) sum[c][e] += __uint_as_float(rc[e]);
          }
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive_cluster(ab == 0 ? acc_empty0 : acc_empty1);
#pragma unroll 1
          for (int h = 0; h < 4; ++h) {
            float x[16];
#pragma unroll
            for (int e = 0; e < 16; ++e) x[e] = sum[0][e];
            emit(x, cc + 16 * h);
#pragma unroll
            for (int e = 0; e < 16; ++e) {
              sum[0][e] = sum[0][16 + e];
              sum[0][16 + e] = sum[1][e];
              sum[1][e] = sum[1][16 + e];
            }
          }
        } else {   // all columns (four epilogue warps): main + cross accumulators
#pragma unroll 1
          for (int ch = 0; ch < kBN / 16; ++ch) {
            uint32_t rm[16], rc[16];
            __syncwarp();
            tmem_ld16_async(acc0 + (uint32_t)(ch * 16), rm);
            tmem_ld16_async(acc0 + (uint32_t)(kBN + ch * 16), rc);
            tmem_ld_wait(rm);
            tmem_ld_wait(rc);
            float x[16];
#pragma unroll
            for (int e = 0; e < 16; ++e) x[e] = __uint_as_float(rm[e]) + __uint_as_float(rc[e]);
            emit(x, ch * 16);
          }
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive_cluster(ab == 0 ? acc_empty0 : acc_empty1);
        }
      } else if (split) {
        // partial Gram product of a split tile: its own fp32 workspace tile
        float* wrow = p.split_ws + (size_t)part_of(t) * (BM * kBN) + (size_t)((int)rank * kHalf + row) * kBN;
#pragma unroll 1
        for (int ch = half0 * (kBN / 64); ch < (half0 + nhalves) * (kBN / 64); ++ch) {
          uint32_t r[32];
          __syncwarp();
          tmem_ld32_async(acc0 + (uint32_t)(ch * 32), r);
          tmem_ld_wait(r);
          const int j0 = t.tn * kBN + ch * 32;
          if (warp_in && j0 < jmax) split_chunk(r, wrow + ch * 32, nscale, i < nrows, ncols - j0);
        }
      } else {
        uint64_t* bf = global_w ? nullptr : box_full;
        // auxbuf: the tile before has been stored (an aux tile: implied by its load)
        if (bf != nullptr && !aux_phase) {
          if (!mbar_wait_warp(box_free, sph ^ 1u, abort_flag, wait_ns)) {
            if (lane == 0) give_up();
            alive = false;
            break;
          }
        }
        if (bf != nullptr) sph ^= 1u;
        const int col0 = t.tn * kBN;
        const int b0 = half0 * (L::kBoxes / 2), bn = (half0 + nhalves) * (L::kBoxes / 2);
        const int b1 = warp_in ? min(bn, max(b0, (jmax - col0) / 64)) : b0;   // boxes inside the padded matrix
        EpiArgs ea;
        ea.i = i;
        ea.nrows = nrows;
        ea.ncols = ncols;
        uint8_t* rowbase = auxbuf + row * 128;
        const int rx = row & 7;
        // warps that reach past the true extent store zeros there
        const bool edge = r0 + 32 > nrows || col0 + 64 * b1 > ncols;
        if (b0 < b1) {
          if (fuse_w_tile) {   // entries past W's extent are not stored (TMA clips them)
            ea.k0 = nscale;
            ea.k1 = fd->shape_scale;
            ea.k2 = p.fuse.eM;
            ea.k3 = p.fuse.lam;
            epi_boxes<kEpiW, false>(acc0, rowbase, rx, b0, b1, col0, ea, bf, lane);
          } else if (phase == NS_POLY) {
            ea.k0 = co.b;
            ea.k1 = co.c;
            ea.k2 = fold ? co.a : 0.f;
            ea.diag = fold ? r0 : -1;
            if (edge) epi_boxes<kEpiPoly, true>(acc0, rowbase, rx, b0, b1, col0, ea, bf, lane);
            else epi_boxes<kEpiPoly, false>(acc0, rowbase, rx, b0, b1, col0, ea, bf, lane);
          } else if (phase == NS_APPLY && !fold) {
            ea.k0 = co.a;
            ea.k1 = kacc;
            ea.k2 = nscale;
            if (edge) epi_boxes<kEpiAxpy, true>(acc0, rowbase, rx, b0, b1, col0, ea, bf, lane);
            else epi_boxes<kEpiAxpy, false>(acc0, rowbase, rx, b0, b1, col0, ea, bf, lane);
          } else {          // GRAM, or X' = B' X
            ea.k0 = nscale;
            if (edge) epi_boxes<kEpiScale, true>(acc0, rowbase, rx, b0, b1, col0, ea, bf, lane);
            else if (nscale != 1.f) epi_boxes<kEpiScale, false>(acc0, rowbase, rx, b0, b1, col0, ea, bf, lane);
            else epi_boxes<kEpiPlain, false>(acc0, rowbase, rx, b0, b1, col0, ea, bf, lane);
          }
        }
        for (int b = b1; bf != nullptr && b < bn; ++b)   // nothing to store there
          if (lane == 0) mbar_arrive(&bf[b]);
      }
      if constexpr (kP == 1) {
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(ab == 0 ? acc_empty0 : acc_empty1);
      }
      if (++ab == kAccRing) {
        ab = 0;
        aph ^= 1u;
      }
      __syncwarp();
      if (kBN == BN && global_w) {
        // Last APPLY: W <- W - eta_M (s X_K + lambda W), with X_K the bf16
        // values just written to auxbuf.  Half-warp h covers row 2k + h of the
        // warp's 32 rows, 16 lanes x 8 columns = 256 contiguous bytes of W.
        for (int half = half0; half < half0 + nhalves; ++half) {
          if (warp_in && write_w) {
            const int cc = lane & 15;
            const int jc = t.tn * BN + half * 128 + cc * 8;
            const unsigned char* box = auxbuf + (2 * half + (cc >> 3)) * kAuxBoxBytes;
            const int ibase = t.tm * BM + (int)rank * kHalf + q * 32 + (lane >> 4);
            __nv_bfloat16* wcol = static_cast<__nv_bfloat16*>(fd->w) + jc;
            for (int k0 = 0; k0 < 16; k0 += kFuseBatch) {
              uint4 wv[kFuseBatch], xv[kFuseBatch];
#pragma unroll
              for (int u = 0; u < kFuseBatch; ++u) {   // all loads of the batch first
                const int rr = q * 32 + 2 * (k0 + u) + (lane >> 4);
                const int ii = ibase + 2 * (k0 + u);
                xv[u] = *reinterpret_cast<const uint4*>(box + rr * 128 + (((cc & 7) ^ (rr & 7)) << 4));
                wv[u] = (ii < nrows && jc < ncols)
                            ? *reinterpret_cast<const uint4*>(wcol + (int64_t)ii * fd->cols)
                            : make_uint4(0u, 0u, 0u, 0u);
              }
#pragma unroll
              for (int u = 0; u < kFuseBatch; ++u) {
                const int ii = ibase + 2 * (k0 + u);
                if (ii >= nrows || jc >= ncols) continue;
                const uint32_t xw[4] = {xv[u].x, xv[u].y, xv[u].z, xv[u].w};
                uint32_t ww[4] = {wv[u].x, wv[u].y, wv[u].z, wv[u].w};
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                  const float w0 = bf_lo(ww[e]), w1 = bf_hi(ww[e]);
                  const float n0 = __fsub_rn(w0, __fmul_rn(p.fuse.eM, __fadd_rn(__fmul_rn(fd->shape_scale, bf_lo(xw[e])),
                                                                               __fmul_rn(p.fuse.lam, w0))));
                  const float n1 = __fsub_rn(w1, __fmul_rn(p.fuse.eM, __fadd_rn(__fmul_rn(fd->shape_scale, bf_hi(xw[e])),
                                                                               __fmul_rn(p.fuse.lam, w1))));
                  ww[e] = pack_bf2(n0, n1);
                }
                *reinterpret_cast<uint4*>(wcol + (int64_t)ii * fd->cols) = make_uint4(ww[0], ww[1], ww[2], ww[3]);
              }
            }
          }
        }
      }
      __syncwarp();
      if (aux_phase) xph ^= 1u;
      // This warp's generic stores are ordered before its count (the reader's
      // proxy fence orders them before its TMA copies).
      if (lane == 0 && global_w) smem_counter_add(aux_left, 1u);
      if (lane == 0 && split) red_release_gpu(p.parts_done + p.part_target[part_of(t)], 1u);
      else if (lane == 0 && kP == 3) red_release_gpu(p.done + 3 * (size_t)(g.first_mat + t.mat) + phase, 1u);
    }
    if (kSplit)
      while (alive && fin_it < fin_end) finish(nullptr, 0u);
  }

  __syncwarp();
  pair_finish<kStages>(*log, abort_flag, full, R.armed, rank);
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, kTmemCols);
  }
}

// Split Gram tiles of the wide kernel: bf16 A tile = the sum of the fp32 parts
// (already scaled), added in part order.
__global__ void __launch_bounds__(256) ns_split_finish_kernel(const NsSplitTarget* __restrict__ targets,
                                                              const float* __restrict__ ws, const unsigned* flags) {
  asm volatile("griddepcontrol.wait;" ::: "memory");   // the Gram launch before it may be programmatic
  if (lm_stopped(flags)) return;
  const NsSplitTarget T = targets[blockIdx.y];
  __nv_bfloat16* dst = static_cast<__nv_bfloat16*>(T.a_tile);
  // four consecutive elements of a row per thread and trip (the tile's
  // column extent is a multiple of 128): 16-byte loads of every part, 8-byte
  // stores; each element's parts are still added in part order
  for (int e = (blockIdx.x * blockDim.x + threadIdx.x) * 4; e < BM * BN; e += gridDim.x * blockDim.x * 4) {
    const int r = e / BN, c = e % BN;
    if (r >= T.nr || c >= T.nc) continue;
    float4 sum = make_float4(0.f, 0.f, 0.f, 0.f);
    const float* part = ws + (size_t)T.first * (BM * BN) + e;
#pragma unroll 4
    for (int k = 0; k < T.nparts; ++k) {
      const float4 v = __ldg(reinterpret_cast<const float4*>(part + (size_t)k * (BM * BN)));
      sum.x += v.x;
      sum.y += v.y;
      sum.z += v.z;
      sum.w += v.w;
    }
    *reinterpret_cast<uint2*>(dst + (size_t)r * T.ld + c) = make_uint2(pack_bf2(sum.x, sum.y), pack_bf2(sum.z, sum.w));
  }
}

// Diagnostic: one thread waits, with the same bounded wait as the NS kernel,
// on an mbarrier nobody arrives on; when the limit passes it records
// LM_FLAG_TIMEOUT and returns normally.
__global__ void bounded_wait_probe_kernel(uint64_t limit_ns, unsigned* flags) {
  __shared__ uint64_t bar;
  __shared__ int abort_flag;
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    if (!mbar_wait(&bar, 0, &abort_flag, limit_ns)) atomicOr(flags, LM_FLAG_TIMEOUT);
  }
}

PFN_cuTensorMapEncodeTiled_v12000 get_encode_fn() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  if (fn == nullptr) {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(f);
  }
  return fn;
}

cudaError_t encode_3d(CUtensorMap* m, void* base, uint64_t inner, uint64_t rows, uint64_t count,
                      uint32_t box_inner, uint32_t box_rows) {
  PFN_cuTensorMapEncodeTiled_v12000 enc = get_encode_fn();
  if (enc == nullptr) return cudaErrorNotSupported;
  const cuuint64_t dims[3] = {inner, rows, count};
  const cuuint64_t strides[2] = {inner * 2, inner * rows * 2};
  const cuuint32_t box[3] = {box_inner, box_rows, 1};
  const cuuint32_t estr[3] = {1, 1, 1};
  CUresult r = enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, base, dims, strides, box, estr,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                   CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

// MN-major operand map: dimensions (64, rows, inner / 64, count), the third
// 128 bytes apart, box (64, box_k, atoms, 1): one copy reads 64 atoms columns.
cudaError_t encode_mn4d(CUtensorMap* m, void* base, uint64_t inner, uint64_t rows, uint64_t count,
                        uint32_t box_k, uint32_t atoms) {
  PFN_cuTensorMapEncodeTiled_v12000 enc = get_encode_fn();
  if (enc == nullptr) return cudaErrorNotSupported;
  const cuuint64_t dims[4] = {64, rows, inner / 64, count};
  const cuuint64_t strides[3] = {inner * 2, 128, inner * rows * 2};
  const cuuint32_t box[4] = {64, box_k, atoms, 1};
  const cuuint32_t estr[4] = {1, 1, 1, 1};
  CUresult r = enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, base, dims, strides, box, estr,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                   CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

}  // namespace

cudaError_t launch_bounded_wait_probe(uint64_t limit_ns, unsigned* flags, cudaStream_t st) {
  count_launch();
  bounded_wait_probe_kernel<<<1, 32, 0, st>>>(limit_ns, flags);
  return cudaGetLastError();
}

cudaError_t tc_encode_w_map(void* w, int64_t rows, int64_t cols, CUtensorMap* map) {
  // W (rows x cols bf16, row-major, cols % 8 = 0, 16-byte aligned) as a 3-D
  // tensor of one matrix, in 64 x 128 boxes
  if (rows <= 0 || cols <= 0 || (cols & 7) != 0 || (reinterpret_cast<uintptr_t>(w) & 15) != 0)
    return cudaErrorInvalidValue;
  return encode_3d(map, w, (uint64_t)cols, (uint64_t)rows, 1, BK, kHalf);
}

int tc_tile_cols(int apply_tiles, int pieces) {
  return pieces == 3 || apply_tiles <= tc_max_pairs() ? 128 : BN;
}
int tc_pad_s(int s) { return (s + kHalf - 1) / kHalf * kHalf; }
int tc_pad_l(int l) { return (l + BN - 1) / BN * BN; }

cudaError_t tc_encode_group_maps(const NsGroup& g, TcGroupMaps* m, int pieces, int bn, bool wide) {
  cudaError_t e = cudaSuccess;
  // three-piece buffers hold piece q of matrix k as matrix k + q * count
  const uint64_t nm = (uint64_t)g.count * (uint64_t)pieces;
  // X buffers: s_pad x l_pad (wide) or l_pad x s_pad (tall), row-major
  const uint64_t inner = g.tall ? g.s_pad : g.l_pad, rows = g.tall ? g.l_pad : g.s_pad;
  auto kmaj = [&](CUtensorMap* map, void* base, uint64_t in, uint64_t r, uint32_t box_rows) {
    if (e == cudaSuccess) e = encode_3d(map, base, in, r, nm, BK, box_rows);
  };
  auto mnmaj = [&](CUtensorMap* map, void* base, uint64_t in, uint64_t r, uint32_t atoms) {
    if (e == cudaSuccess) e = encode_mn4d(map, base, in, r, nm, BK, atoms);
  };
  for (int b = 0; b < 2; ++b) {
    kmaj(&m->xk[b], g.X[b], inner, rows, kHalf);
    mnmaj(&m->xmn[b], g.X[b], inner, rows, 2);
  }
  kmaj(&m->a, g.A, g.s_pad, g.s_pad, kHalf);
  kmaj(&m->b, g.B, g.s_pad, g.s_pad, kHalf);
  mnmaj(&m->amn, g.A, g.s_pad, g.s_pad, 2);
  mnmaj(&m->bmn, g.B, g.s_pad, g.s_pad, 2);
  if (bn == BN) {   // a CTA's B rows are a 128-wide half, as its A rows
    for (int b = 0; b < 2; ++b) {
      m->nxk[b] = m->xk[b];
      m->nxmn[b] = m->xmn[b];
    }
    m->na = m->a;
    m->nb = m->b;
    m->namn = m->amn;
    m->nbmn = m->bmn;
  } else {
    for (int b = 0; b < 2; ++b) {
      kmaj(&m->nxk[b], g.X[b], inner, rows, (uint32_t)bn / 2);
      mnmaj(&m->nxmn[b], g.X[b], inner, rows, (uint32_t)bn / 128);
    }
    kmaj(&m->na, g.A, g.s_pad, g.s_pad, (uint32_t)bn / 2);
    kmaj(&m->nb, g.B, g.s_pad, g.s_pad, (uint32_t)bn / 2);
    mnmaj(&m->namn, g.A, g.s_pad, g.s_pad, (uint32_t)bn / 128);
    mnmaj(&m->nbmn, g.B, g.s_pad, g.s_pad, (uint32_t)bn / 128);
  }
  if (wide) {   // the wide kernel stores 32-row boxes per warp
    for (int b = 0; b < 2; ++b)
      if (e == cudaSuccess) e = encode_3d(&m->xst[b], g.X[b], inner, rows, nm, 64, 32);
    if (e == cudaSuccess) e = encode_3d(&m->ast, g.A, g.s_pad, g.s_pad, nm, 64, 32);
    if (e == cudaSuccess) e = encode_3d(&m->bst, g.B, g.s_pad, g.s_pad, nm, 64, 32);
  }
  return e;
}

namespace {
__global__ void __launch_bounds__(256) split3_kernel(const float4* __restrict__ src, uint2* __restrict__ dst,
                                                     size_t n4, const unsigned* flags) {
  if (lm_stopped(flags)) return;
  for (size_t k = blockIdx.x * (size_t)blockDim.x + threadIdx.x; k < n4; k += (size_t)gridDim.x * blockDim.x) {
    const float4 v = src[k];
    float h[4], m[4], l[4];
    split3(v.x, h[0], m[0], l[0]);
    split3(v.y, h[1], m[1], l[1]);
    split3(v.z, h[2], m[2], l[2]);
    split3(v.w, h[3], m[3], l[3]);
    dst[k] = make_uint2(pack_bf2(h[0], h[1]), pack_bf2(h[2], h[3]));
    dst[n4 + k] = make_uint2(pack_bf2(m[0], m[1]), pack_bf2(m[2], m[3]));
    dst[2 * n4 + k] = make_uint2(pack_bf2(l[0], l[1]), pack_bf2(l[2], l[3]));
  }
}
}  // namespace

cudaError_t launch_split3(const float* src, void* dst, size_t n, const unsigned* flags, cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  if (n % 4 != 0) return cudaErrorInvalidValue;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const size_t n4 = n / 4;
  size_t grid = (n4 + 255) / 256;
  if (grid > (size_t)sms * 8) grid = (size_t)sms * 8;
  count_launch();
  split3_kernel<<<(unsigned)grid, 256, 0, st>>>(reinterpret_cast<const float4*>(src), static_cast<uint2*>(dst), n4, flags);
  return cudaGetLastError();
}

cudaError_t launch_ns_split_finish(const NsSplitTarget* targets, int n, const float* ws, const unsigned* flags,
                                   cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  count_launch();
  ns_split_finish_kernel<<<dim3(32, n), 256, 0, st>>>(targets, ws, flags);
  return cudaGetLastError();
}

template <bool kSplit, int kP, int kBN, bool kPromo = false>
static cudaError_t set_smem_attr() {
  return cudaFuncSetAttribute(ns_tc_kernel<kSplit, kP, kBN, kPromo>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)TcLayout<kP, kBN>::kSmemBytes);
}

// Whether launches on st run on a part of the device's SMs only (a stream of a
// green context; a stream that cannot be asked is taken for one).
static bool part_of_device(cudaStream_t st) {
  static const PFN_cuStreamGetCtx_v12050 get = []() -> PFN_cuStreamGetCtx_v12050 {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuStreamGetCtx", &f, 12050, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      return reinterpret_cast<PFN_cuStreamGetCtx_v12050>(f);
    return nullptr;
  }();
  CUcontext ctx = nullptr;
  CUgreenCtx green = nullptr;
  return get == nullptr || get(st, &ctx, &green) != CUDA_SUCCESS || green != nullptr;
}

template <bool kSplit, int kP, int kBN, bool kPromo = false>
static cudaError_t launch_chain(const ChainParams& prm, int grid, bool together, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid, 1, 1);
  cfg.blockDim = dim3(kChainThreads, 1, 1);
  cfg.dynamicSmemBytes = TcLayout<kP, kBN>::kSmemBytes;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;   // (together) pairs wait for one another: all resident or none
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = together ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, ns_tc_kernel<kSplit, kP, kBN, kPromo>, prm);
}

int tc_max_pairs() {
  static int cached[kMaxDevices] = {};
  const int slot = device_slot();
  if (slot >= 0 && cached[slot] > 0) return cached[slot];
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  int pairs = sms / 2 > 0 ? sms / 2 : 1;
  // (planned for the whole device, also from within a part of it)
  if (sms > 0 && part_of_device(nullptr)) return pairs;
  // the pairs of a chain launch must all be resident at once
  if (set_smem_attr<true, 1, 256>() == cudaSuccess) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(2 * pairs), 1, 1);
    cfg.blockDim = dim3(kChainThreads, 1, 1);
    cfg.dynamicSmemBytes = TcLayout<1, 256>::kSmemBytes;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, ns_tc_kernel<true, 1, 256, false>, &cfg) == cudaSuccess && n > 0 && n < pairs) pairs = n;
  }
  cudaGetLastError();   // no device (planning on the host alone): not an error here
  if (slot >= 0) cached[slot] = pairs;
  return pairs;
}

// What a launch runs of its phases: tiles and the sums of split Gram targets,
// or one of the two.
enum ChainPart { kTilesAndSums, kTilesOnly, kSumsOnly };
static cudaError_t launch_chain_part(const NsChain& c, int q0, int q1, ChainPart part, bool together, cudaStream_t st) {
  if (q0 >= q1) return cudaSuccess;
  if (c.ngroups < 1 || c.ngroups > kMaxGroupsTc || c.steps < 1 || c.steps > kMaxNsSteps || c.npairs < 1 ||
      (c.pieces != 1 && c.pieces != 3) || (c.pieces == 3 && c.fuse != nullptr) || c.wait_ns == 0 ||
      (c.bn != 256 && c.bn != 128) || (c.pieces == 3 && c.bn != 128))
    return cudaErrorInvalidValue;
  static bool attr_set[kMaxDevices] = {};
  const int slot = device_slot();
  if (slot < 0 || !attr_set[slot]) {
    cudaError_t e = set_smem_attr<false, 1, 256>();
    if (e == cudaSuccess) e = set_smem_attr<true, 1, 256>();
    if (e == cudaSuccess) e = set_smem_attr<false, 1, 128>();
    if (e == cudaSuccess) e = set_smem_attr<true, 1, 128>();
    if (e == cudaSuccess) e = set_smem_attr<false, 3, 128>();
    if (e == cudaSuccess) e = set_smem_attr<true, 3, 128>();
    if (e == cudaSuccess) e = set_smem_attr<false, 3, 128, true>();
    if (e == cudaSuccess) e = set_smem_attr<true, 3, 128, true>();
    if (e != cudaSuccess) return e;
    if (slot >= 0) attr_set[slot] = true;
  }
  ChainParams prm;
  memset(&prm, 0, sizeof(prm));
  for (int gi = 0; gi < c.ngroups; ++gi) {
    prm.maps[gi] = c.maps[gi];
    prm.groups[gi] = c.groups[gi];
  }
  for (int ph = 0; ph < 3; ++ph) {
    prm.tiles[ph] = c.tiles[ph];
    prm.offsets[ph] = c.offsets[ph];
    prm.ntiles[ph] = c.ntiles[ph];
  }
  prm.counts = c.counts;
  prm.targets = c.targets;
  prm.part_target = c.part_target;
  prm.ntargets = c.ntargets;
  prm.split_ws = c.split_ws;
  prm.parts_done = c.parts_done;
  prm.done = c.done;
  prm.norm2 = c.norm2;
  prm.q0 = q0;
  prm.q1 = q1;
  prm.steps = c.steps;
  prm.flags = c.flags;
  prm.active = c.active;
  prm.wait_ns = c.wait_ns;
  uint32_t npoly = 0;
  for (int it = 0; it < c.steps; ++it) {
    const NsCoeffs& co = c.co[it];
    prm.eps = co.eps;
    const NsIterForm f = ns_iter_form(co, c.pieces, c.fold);
    npoly += f.from_a ? 0u : 1u;
    prm.it[it] = ChainIter{co.a, co.b, co.c, (f.from_a ? kIterFromA : 0u) | (f.fold ? kIterFold : 0u) | (npoly << 8)};
  }
  // epilogue warps that signal: four (with register sums eight, half the columns
  // each); the parameter write that reads W from
  // global memory (last APPLY, a not folded) has a launch of its own with eight
  const bool last_fused = c.fuse != nullptr && q1 == 3 * c.steps;
  const bool global_w = last_fused && !(prm.it[c.steps - 1].mode & kIterFold);
  if (global_w && c.bn != 256) return cudaErrorInvalidValue;
  if (global_w && q0 != 3 * c.steps - 1) {
    cudaError_t e = launch_chain_part(c, q0, q1 - 1, part, together, st);
    return e == cudaSuccess ? launch_chain_part(c, q1 - 1, q1, part, together, st) : e;
  }
  if (last_fused) prm.fuse = *c.fuse;
  const int base_epi = c.pieces == 3 && c.promote ? kEpiWarps : 4;
  prm.nepi = global_w ? kEpiWarps : base_epi;
  prm.part_sig = 2u * (uint32_t)base_epi;
  prm.sig = c.pieces == 1 ? 2u : prm.part_sig;
  // about one finish unit per epilogue warp, 4 to 32 rows each
  const int warps = 2 * c.npairs * kEpiWarps;
  prm.fin_units = 8;
  while (prm.fin_units < 64 && prm.fin_units * c.ntargets * 2 <= warps) prm.fin_units *= 2;
  if (part == kTilesOnly) prm.ntargets = 0;
  for (int ph = 0; ph < 3 && part == kSumsOnly; ++ph) {
    prm.offsets[ph] = nullptr;
    prm.ntiles[ph] = 0;
    prm.counts = nullptr;
  }
  const int grid = 2 * c.npairs;
  const bool split = c.ntargets > 0;
  count_launch();
  if (c.pieces == 3 && c.promote)
    return split ? launch_chain<true, 3, 128, true>(prm, grid, together, st)
                 : launch_chain<false, 3, 128, true>(prm, grid, together, st);
  if (c.pieces == 3)
    return split ? launch_chain<true, 3, 128>(prm, grid, together, st)
                 : launch_chain<false, 3, 128>(prm, grid, together, st);
  if (c.bn == 128)
    return split ? launch_chain<true, 1, 128>(prm, grid, together, st)
                 : launch_chain<false, 1, 128>(prm, grid, together, st);
  return split ? launch_chain<true, 1, 256>(prm, grid, together, st)
               : launch_chain<false, 1, 256>(prm, grid, together, st);
}

// On a part of the device the planned pairs may not all be resident, and no
// launch may wait for another pair: one launch per phase, and one more for the
// sums of a phase's split Gram targets, neither cooperative (a cooperative
// launch larger than the part does not return).  Then every counter a launch
// waits for was reached by the launches before it.
cudaError_t launch_ns_chain(const NsChain& c, int q0, int q1, cudaStream_t st) {
  if (!part_of_device(st)) return launch_chain_part(c, q0, q1, kTilesAndSums, true, st);
  for (int q = q0; q < q1; ++q) {
    if (q % 3 == NS_POLY && ns_iter_form(c.co[q / 3], c.pieces, c.fold).from_a) continue;
    cudaError_t e = launch_chain_part(c, q, q + 1, kTilesOnly, false, st);
    if (e == cudaSuccess && q % 3 == NS_GRAM && c.ntargets > 0)
      e = launch_chain_part(c, q, q + 1, kSumsOnly, false, st);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t launch_ns_wide_phase(NsPhase ph, int iter, int ngroups, const NsGroup* groups, const TcGroupMaps* maps,
                                 const NsTile* tiles, int ntiles, const int* offsets, int npairs,
                                 const double* norm2, NsCoeffs co, unsigned* flags, const FuseFinal* fuse,
                                 cudaStream_t st, const unsigned char* active, float* split_ws, bool pdl,
                                 uint64_t wait_ns) {
  if (ntiles <= 0) return cudaSuccess;
  if (ngroups < 1 || ngroups > kMaxGroupsTc || wait_ns == 0) return cudaErrorInvalidValue;
  TcParams prm;
  memset(&prm, 0, sizeof(prm));
  for (int gi = 0; gi < ngroups; ++gi) {
    prm.maps[gi] = maps[gi];
    prm.groups[gi] = groups[gi];
  }
  prm.tiles = tiles;
  prm.offsets = offsets;
  prm.ntiles = ntiles;
  prm.phase = (int)ph;
  prm.iter = iter;
  prm.norm2 = norm2;
  prm.co = co;
  prm.flags = flags;
  if (fuse != nullptr && ph == NS_APPLY) prm.fuse = *fuse;
  prm.active = active;
  prm.split_ws = split_ws;
  prm.wait_ns = wait_ns;
  const bool split = split_ws != nullptr && ph == NS_GRAM;
  return launch_ns_wide(prm, 2 * npairs, active != nullptr, split, pdl, st);
}

// Active tiles of a masked step, in list order: block ph compacts the tiles of
// phase ph whose matrix is selected and writes their count.
namespace {
struct CompactArgs {
  const NsTile* src[3];
  NsTile* dst[3];
  int n[3];
  int* counts;
  const NsGroup* groups;
  const unsigned char* active;
  const unsigned* flags;
};
__global__ void __launch_bounds__(1024) ns_compact_kernel(const __grid_constant__ CompactArgs a) {
  __shared__ int warp_sum[32];
  __shared__ int base;
  const int ph = blockIdx.x, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (lm_stopped(a.flags)) {   // the chain launch will stop as well
    if (tid == 0) a.counts[ph] = 0;
    return;
  }
  if (tid == 0) base = 0;
  __syncthreads();
  for (int k0 = 0; k0 < a.n[ph]; k0 += 1024) {
    const int k = k0 + tid;
    NsTile t{};
    bool on = false;
    if (k < a.n[ph]) {
      t = a.src[ph][k];
      on = a.active[a.groups[t.group].first_mat + t.mat] != 0;
    }
    const unsigned m = __ballot_sync(0xffffffffu, on);
    if (lane == 0) warp_sum[warp] = __popc(m);
    __syncthreads();
    int before = base;
    for (int w = 0; w < warp; ++w) before += warp_sum[w];
    if (on) a.dst[ph][before + __popc(m & ((1u << lane) - 1u))] = t;
    __syncthreads();
    if (tid == 1023) base = before + __popc(m);
    __syncthreads();
  }
  if (tid == 0) a.counts[ph] = base;
}
}  // namespace

cudaError_t launch_ns_compact(const NsTile* const* src, NsTile* const* dst, const int* n, int* counts,
                              const NsGroup* groups, const unsigned char* active, const unsigned* flags,
                              cudaStream_t st) {
  CompactArgs a;
  for (int ph = 0; ph < 3; ++ph) {
    a.src[ph] = src[ph];
    a.dst[ph] = dst[ph];
    a.n[ph] = n[ph];
  }
  a.counts = counts;
  a.groups = groups;
  a.active = active;
  a.flags = flags;
  count_launch();
  ns_compact_kernel<<<3, 1024, 0, st>>>(a);
  return cudaGetLastError();
}

}  // namespace lm
