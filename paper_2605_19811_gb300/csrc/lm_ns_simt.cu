// fp32 CUDA-core Newton-Schulz phases (the "fp32 mode" of the msign
// approximation; Section 2 names the odd-polynomial iteration).  Per
// iteration, for every matrix X of every group (s x l, or l x s for a tall
// parameter, which iterates on X^T X and X B instead):
//   GRAM : A = X X^T          (tiles on or above the diagonal, mirrored store)
//   POLY : B = b A + c A A    (tiles on or above the diagonal, mirrored store)
//   APPLY: X' = a X + B X
// Iteration 0 folds the normalisation X / (||G_hat||_F + eps) into GRAM
// (scale 1/(n+eps)^2) and APPLY (scale 1/(n+eps)).  Sets with small matrices
// run here (f32_on_tensor_cores says which), sets whose three-piece workspace
// does not fit the device, and lm_msign_ns_noalloc.
//
// A block of 256 threads computes one square tile: 128 x 128 (8 x 8 outputs per
// thread in 4 x 4 quadrants 64 apart, K slices of 16, two blocks per SM) or 64 x
// 64 (4 x 4 outputs, K slices of 32, four blocks per SM).  Slices are double-
// buffered in shared memory: the global loads of slice k + 1 are in flight
// while slice k is multiplied.
// A phase that would leave more than a fifth of the resident 128-wide blocks,
// over all its rounds, without work takes 64-wide ones, and where those leave
// blocks idle too, tiles are cut along K: each part writes its partial tile, and
// the block that finishes last adds the parts in order and writes the result,
// so the sum does not depend on timing and nothing waits.
// Same box, against 128-wide tiles only and a summing launch after each split
// Gram: tiny fp32 set (256 x 256 to 256 x 1024, which now runs on the tensor
// cores) 541 -> 314 us per Muon step, msign of 1024 x 1024 1497 -> 1026 us,
// lm_msign_ns_noalloc of 1024 x 1024 1795 -> 917 us.
#include "lm_internal.h"

namespace lm {
namespace {

constexpr int kThreads = 256;
constexpr int kPadS = 4;   // row padding of the shared tiles (floats)

// One kTile (i) x BK (k) operand slice, two float4 per thread, from a K-major
// (element (i, k) at op[i * ld + k]) or MN-major (at op[k * ld + i]) matrix.
// 64-wide: a warp reads 8 rows x 64 bytes of a K-major one, so that its
// transposed stores meet at most two to a bank.
struct SliceRegs {
  float4 v[2];
};
template <int kTile>
__device__ __forceinline__ void slice_at(int u, bool mn, int& i, int& k) {
  const int t = threadIdx.x, f = t + u * kThreads;
  if (mn) {
    i = f % (kTile / 4) * 4;
    k = f / (kTile / 4);
  } else if (kTile == 128) {
    i = f >> 2;
    k = (f & 3) * 4;
  } else {
    i = (t & 7) | ((t >> 5) << 3);
    k = ((t >> 3) & 3) * 4 + 16 * u;
  }
}
template <int kTile>
__device__ __forceinline__ void load_slice(SliceRegs& R, const float* op, int ld, bool mn, int i0, int k0) {
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    int i, k;
    slice_at<kTile>(u, mn, i, k);
    if (!mn) R.v[u] = *reinterpret_cast<const float4*>(op + (size_t)(i0 + i) * ld + k0 + k);
    else R.v[u] = *reinterpret_cast<const float4*>(op + (size_t)(k0 + k) * ld + i0 + i);
  }
}
template <int kTile>
__device__ __forceinline__ void store_slice(float (*S)[kTile + kPadS], const SliceRegs& R, bool mn) {
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    int i, k;
    slice_at<kTile>(u, mn, i, k);
    if (!mn) {
      S[k + 0][i] = R.v[u].x; S[k + 1][i] = R.v[u].y; S[k + 2][i] = R.v[u].z; S[k + 3][i] = R.v[u].w;
    } else {
      *reinterpret_cast<float4*>(&S[k][i]) = R.v[u];
    }
  }
}

// Wide groups hold X as s x l, tall groups as l x s:
//   GRAM  wide A = X X^T (rows of X), tall A = X^T X (columns of X)
//   POLY  B = b A + c A A
//   APPLY wide X' = a X + B X, tall X' = a X + X B
// A and B are kept whole, so their rows serve as columns: POLY and the left
// operand of the wide APPLY read them MN-major (no transposed stores).
template <int kTile, bool kSplit>
__global__ void __launch_bounds__(kThreads, kTile == 128 ? 2 : 4)
    ns_simt_kernel(int phase, int iter, const NsGroup* __restrict__ groups,
                   const NsTile* __restrict__ tiles, int ntiles, const double* __restrict__ norm2,
                   NsCoeffs co, const unsigned char* __restrict__ active, float* split_ws,
                   uint32_t* parts_done, const unsigned* flags) {
  constexpr int BK = simt_slice(kTile), Q = kTile / 64, T = 4 * Q, H = 64;   // Q x Q quadrants H apart
  if (lm_stopped(flags)) return;
  __shared__ __align__(16) float As[2][BK][kTile + kPadS];
  __shared__ __align__(16) float Bs[2][BK][kTile + kPadS];
  __shared__ int last_part;
  const int tid = threadIdx.x;
  const int tx = kTile == 128 ? tid & 15 : (tid & 7) | ((tid >> 2) & 8);   // 64-wide: a warp stands 8 x 4
  const int ty = kTile == 128 ? tid >> 4 : ((tid >> 3) & 3) | ((tid >> 6) << 2);

  for (int w = blockIdx.x; w < ntiles; w += gridDim.x) {
    const NsTile t = tiles[w];
    const NsGroup& g = groups[t.group];
    if (active != nullptr && !active[g.first_mat + t.mat]) continue;   // block-uniform
    const int cur = iter & 1;
    const bool tall = g.tall != 0;
    const int ldx = tall ? g.s_pad : g.l_pad;
    const float* X = static_cast<const float*>(cur ? g.X[1] : g.X[0]) + (size_t)t.mat * g.s_pad * g.l_pad;
    const float* Am = static_cast<const float*>(g.A) + (size_t)t.mat * g.s_pad * g.s_pad;
    const float* Bm = static_cast<const float*>(g.B) + (size_t)t.mat * g.s_pad * g.s_pad;
    const float* opA;
    const float* opB;
    int lda, ldb, K;
    bool amn, bmn;
    if (phase == NS_GRAM) {
      opA = X; opB = X; lda = ldb = ldx; K = g.l_pad; amn = bmn = tall;
    } else if (phase == NS_POLY) {
      opA = Am; opB = Am; lda = ldb = g.s_pad; K = g.s_pad; amn = bmn = true;
    } else if (tall) {
      opA = X; opB = Bm; lda = ldx; ldb = g.s_pad; K = g.s_pad; amn = false; bmn = true;
    } else {
      opA = Bm; opB = X; lda = g.s_pad; ldb = ldx; K = g.s_pad; amn = bmn = true;
    }
    const int i0 = t.tm * kTile, j0 = t.tn * kTile;
    const bool split = kSplit && t.slot != 0;   // K slices [kb0, kb1) of the tile
    const int kbeg = split ? (int)t.kb0 * BK : 0;
    const int kend = split ? (int)t.kb1 * BK : K;
    float acc[T][T];
#pragma unroll
    for (int a = 0; a < T; ++a)
#pragma unroll
      for (int b = 0; b < T; ++b) acc[a][b] = 0.f;

    SliceRegs ra, rb;
    load_slice<kTile>(ra, opA, lda, amn, i0, kbeg);
    load_slice<kTile>(rb, opB, ldb, bmn, j0, kbeg);
    __syncthreads();   // the previous tile's last reads of the buffers are done
    store_slice<kTile>(As[0], ra, amn);
    store_slice<kTile>(Bs[0], rb, bmn);
    __syncthreads();
    int buf = 0;
    for (int k0 = kbeg; k0 < kend; k0 += BK) {
      const bool more = k0 + BK < kend;
      if (more) {   // next slice in flight while this one is multiplied
        load_slice<kTile>(ra, opA, lda, amn, i0, k0 + BK);
        load_slice<kTile>(rb, opB, ldb, bmn, j0, k0 + BK);
      }
#pragma unroll
      for (int kk = 0; kk < BK; ++kk) {
        float av[T], bv[T];
#pragma unroll
        for (int q = 0; q < Q; ++q) {
          const float4 a4 = *reinterpret_cast<const float4*>(&As[buf][kk][H * q + ty * 4]);
          const float4 b4 = *reinterpret_cast<const float4*>(&Bs[buf][kk][H * q + tx * 4]);
          av[4 * q] = a4.x; av[4 * q + 1] = a4.y; av[4 * q + 2] = a4.z; av[4 * q + 3] = a4.w;
          bv[4 * q] = b4.x; bv[4 * q + 1] = b4.y; bv[4 * q + 2] = b4.z; bv[4 * q + 3] = b4.w;
        }
#pragma unroll
        for (int a = 0; a < T; ++a)
#pragma unroll
          for (int b = 0; b < T; ++b) acc[a][b] = fmaf(av[a], bv[b], acc[a][b]);
      }
      if (more) {
        store_slice<kTile>(As[buf ^ 1], ra, amn);
        store_slice<kTile>(Bs[buf ^ 1], rb, bmn);
        __syncthreads();
        buf ^= 1;
      }
    }

    if constexpr (kSplit) if (split) {
      // this part's tile, 16 bytes per thread and row; the last part to get
      // here (nh: part index << 8 | parts) adds all of them in part order
      const int part = t.nh >> 8, nparts = t.nh & 255, first = (int)t.slot - 1 - part;
      float* ws = split_ws + (size_t)(t.slot - 1) * (kTile * kTile);
#pragma unroll
      for (int a = 0; a < T; ++a)
#pragma unroll
        for (int q = 0; q < Q; ++q)
          __stcg(reinterpret_cast<float4*>(ws + (size_t)((a >> 2) * H + ty * 4 + (a & 3)) * kTile + H * q + tx * 4),
                 make_float4(acc[a][4 * q], acc[a][4 * q + 1], acc[a][4 * q + 2], acc[a][4 * q + 3]));
      __threadfence();
      __syncthreads();
      if (tid == 0) {
        const uint32_t before = atomicAdd(parts_done + first, 1u);
        last_part = before == (uint32_t)nparts - 1u ? 1 : 0;
        if (last_part) parts_done[first] = 0u;   // for the next launch
      }
      __syncthreads();
      if (!last_part) continue;
      __threadfence();
      const float* src = split_ws + (size_t)first * (kTile * kTile);
#pragma unroll
      for (int a = 0; a < T; ++a)
#pragma unroll
        for (int q = 0; q < Q; ++q) {
          const size_t o = (size_t)((a >> 2) * H + ty * 4 + (a & 3)) * kTile + H * q + tx * 4;
          float4 sum = __ldcg(reinterpret_cast<const float4*>(src + o));
          for (int k = 1; k < nparts; ++k) {
            const float4 v = __ldcg(reinterpret_cast<const float4*>(src + (size_t)k * (kTile * kTile) + o));
            sum.x += v.x;
            sum.y += v.y;
            sum.z += v.z;
            sum.w += v.w;
          }
          acc[a][4 * q] = sum.x; acc[a][4 * q + 1] = sum.y; acc[a][4 * q + 2] = sum.z; acc[a][4 * q + 3] = sum.w;
        }
    }

    // epilogue: rows i0 + ty*4 + a (+ H), columns j0 + tx*4 + b (+ H).  A
    // diagonal tile holds both halves (equal: the same products in the same
    // order); a tile above the diagonal also stores its mirror.
    float nscale = 1.f;
    if (iter == 0) {
      const float n = (float)sqrt(norm2[g.first_mat + t.mat]) + co.eps;
      nscale = (phase == NS_GRAM) ? 1.f / (n * n) : (phase == NS_APPLY ? 1.f / n : 1.f);
    }
    const int nrows = (phase == NS_APPLY && tall) ? g.l : g.s;
    const int ncols = (phase == NS_APPLY) ? (tall ? g.s : g.l) : g.s;
    const int ldo = phase == NS_APPLY ? ldx : g.s_pad;
    float* out = phase == NS_GRAM ? const_cast<float*>(Am)
               : phase == NS_POLY ? const_cast<float*>(Bm)
                                  : static_cast<float*>(cur ? g.X[0] : g.X[1]) + (size_t)t.mat * g.s_pad * g.l_pad;
    const float* aux = phase == NS_POLY ? Am : X;
#pragma unroll
    for (int qa = 0; qa < Q; ++qa)
#pragma unroll
      for (int q = 0; q < Q; ++q) {
        const int ib = i0 + H * qa + ty * 4, jb = j0 + H * q + tx * 4;
        float o[4][4];
#pragma unroll
        for (int a = 0; a < 4; ++a) {
          const int i = ib + a;
          float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
          if (phase != NS_GRAM) x = *reinterpret_cast<const float4*>(aux + (size_t)i * ldo + jb);
          const float xv[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
          for (int b = 0; b < 4; ++b) {
            const float c = acc[4 * qa + a][4 * q + b];
            const float v = phase == NS_GRAM ? c * nscale
                          : phase == NS_POLY ? co.b * xv[b] + co.c * c
                                             : (co.a * xv[b] + c) * nscale;
            o[a][b] = i < nrows && jb + b < ncols ? v : 0.f;
          }
          *reinterpret_cast<float4*>(out + (size_t)i * ldo + jb) = make_float4(o[a][0], o[a][1], o[a][2], o[a][3]);
        }
        if (phase != NS_APPLY && t.tm != t.tn) {
#pragma unroll
          for (int b = 0; b < 4; ++b)
            *reinterpret_cast<float4*>(out + (size_t)(jb + b) * ldo + ib) =
                make_float4(o[0][b], o[1][b], o[2][b], o[3][b]);
        }
      }
  }
}

}  // namespace

int simt_pad(int x) { return (x + kSimtBM - 1) / kSimtBM * kSimtBM; }

int simt_blocks(int tile, int sms) { return (tile == 128 ? 2 : 4) * (sms > 0 ? sms : 1); }

int simt_tile(int64_t tiles128, int sms) {
  const int64_t slots = simt_blocks(128, sms), rounds = (tiles128 + slots - 1) / slots;
  return 5 * tiles128 < 4 * rounds * slots ? 64 : 128;
}

cudaError_t launch_ns_simt(NsPhase ph, int iter, int tile, const NsGroup* dgroups, const NsTile* tiles, int ntiles,
                           const double* norm2, NsCoeffs co, cudaStream_t st, const unsigned char* active,
                           float* split_ws, uint32_t* parts_done, const unsigned* flags) {
  if (ntiles <= 0) return cudaSuccess;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int slots = simt_blocks(tile, sms);
  const int grid = ntiles < slots ? ntiles : slots;
  count_launch();
  const bool split = split_ws != nullptr;
  auto kern = tile == 128 ? (split ? ns_simt_kernel<128, true> : ns_simt_kernel<128, false>)
                          : (split ? ns_simt_kernel<64, true> : ns_simt_kernel<64, false>);
  kern<<<grid, kThreads, 0, st>>>((int)ph, iter, dgroups, tiles, ntiles, norm2, co, active, split_ws, parts_done, flags);
  return cudaGetLastError();
}

}  // namespace lm
