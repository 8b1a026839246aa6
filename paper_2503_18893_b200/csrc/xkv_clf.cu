// Cross-layer factorisation on the GPU (Sec. 3.1, Eq. 1; App. "Custom SVD Kernel": a randomised SVD whose power
// iterations are 16-bit tensor-core matrix products and whose orthogonalisation is a shifted Cholesky QR).
//
// X = [X_l0 ... X_l0+G-1] (T x N, N = G d, bf16) is tall, so the iteration runs on the right side.  With l = r + p:
//   Z (N x l) <- the random test matrix
//   repeat q + 1 times:   Y^T = Z^T X^T   (l x T, bf16)          tensor core
//                         U   = X^T Y     (N x l, fp32)          tensor core
//                         Z   = U R^-1,  R^T R = U^T U + shift I (shifted Cholesky QR in fp64: one pass inside the
//                               iteration, three for the last iterate, which has to be orthonormal)
//   Rayleigh-Ritz:        W^T = Z^T X^T,  M = W^T W (= Z^T X^T X Z, l x l),  M = P Lambda P^T (Jacobi); Z and W as sums of
//                         two bf16 matrices here
//   V = Z P_r (N x r);    B_l = rows of V^T (bf16);   A = X V = W P_r (T x r, tensor core);   sigma = sqrt(Lambda).
// A = U Sigma and B = V^T of the truncated SVD of X, up to the accuracy of the subspace (checked against the exact
// optimum sum_{i>r} sigma_i^2, never factor by factor: signs and degenerate subspaces are not unique).
//
// One tensor-core kernel serves the tall products.  It computes C (M x N) = A B with either operand K-major (its rows run
// along k) or MN-major (its rows run along m or n), which the shared-memory descriptors cover, so no matrix is ever
// transposed in memory:
//   Y = X Z (X K-major, Z MN-major), stored transposed as Y^T;    U = X^T Y (X MN-major, Y^T K-major);
//   M = W^T W (W^T K-major twice);                                 A = W P (W^T MN-major, P^T K-major) or
//                                                                  A = X V (X K-major, V MN-major).
#include <cuda.h>
#include <math.h>

#include "xkv_internal.cuh"
#include "xkv_ptx.cuh"

namespace xkv {

namespace {

using namespace ptx;

// Tiles are (128 MB) x BN, MB accumulators of 128 rows in tensor memory sharing the B operand; one stage of the operand
// ring holds 64 k.  What bounds the products is the rate at which L2 feeds the SMs (about 53 bytes per cycle and SM when
// all of them ask): a 128 x 256 tile wants 96, a 256 x 192 tile 73 and a 256 x 256 tile 64 at the full rate of the tensor
// core.  X Z at 131072 x 4096 x 576, a CTA per tile: 0.87 ms with 128 x 256 tiles, 0.50 with 256 x 192;
// X^T Y 0.65 ms with 96 tiles of 128 x 192, 0.40 with 48 of 256 x 192 over three K ranges.
constexpr int kGemmEpiWarps = 4;                  // per 128 rows; then one TMA producer warp, one MMA issue warp
template <int MB> constexpr int gemm_threads() { return (MB * kGemmEpiWarps + 2) * 32; }
template <int MB, int BN> constexpr int gemm_stage_bytes() { return MB * 16384 + BN * 128; }
template <int MB, int BN> constexpr int gemm_stages() { return MB == 2 && BN == 256 ? 3 : MB == 1 && BN == 128 ? 3 : 4; }
constexpr int kGemmMaxStages = 4;
constexpr uint32_t kGemmWaitLimit = 1u << 24;

__device__ __forceinline__ bool gemm_wait(uint32_t bar, uint32_t parity) {
  for (uint32_t i = 0; i < kGemmWaitLimit; ++i) {
    if (mbar_try_wait(bar, parity)) return true;
  }
  return false;
}

// C[m][n] = sum_k A(k, m) B(k, n).  tiles = (ceil(N/BN), ceil(M/(128 MB)), K ranges), the first fastest; a CTA takes every
// gridDim.x-th of them.  The operand ring runs on from tile to tile, and a result in bf16 alone leaves tensor memory for
// registers before it is stored, so that the next tile's products run beside its stores.  131072 x 4096 x 576: 495 us with a
// CTA per tile, 421 now; with two parts of B and of the result 930 -> 855.
// TRANS: store C^T (out[n][m]).
// AK: A is given as [m][k] (K-major), else as [k][m]; BK likewise for B.  K range z covers k_per columns and writes
// Cf + z * M * ldc.  With two parts B is the sum of the matrices of map_b and map_b2 and A is gone through twice, a third
// adds the product of those of map_a3 and map_b3; the k of a part are rounded up to whole blocks of 64.  Cb is the result rounded to bf16; LO: Cl is twice what the rounding leaves
// out (TRANS only; a template parameter, because a test of the pointer in the epilogue costs every product 11 %).  Out-of-range rows and columns of the operands are zero-filled by the copy engine; stores are guarded.
template <bool TRANS, bool AK, bool BK, bool LO, int MB, int BN>
__global__ void __launch_bounds__(gemm_threads<MB>(), 1)
clf_gemm_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b,
                const __grid_constant__ CUtensorMap map_b2, const __grid_constant__ CUtensorMap map_a3,
                const __grid_constant__ CUtensorMap map_b3, int M, int N, int k_part, int k_all, int k_per, float* __restrict__ Cf,
                __nv_bfloat16* __restrict__ Cb, __nv_bfloat16* __restrict__ Cl, long long ldc, dim3 tiles, unsigned int* __restrict__ flags) {
  extern __shared__ uint8_t gemm_smem[];
  constexpr int kGemmStages = gemm_stages<MB, BN>(), kGemmStageBytes = gemm_stage_bytes<MB, BN>();
  constexpr uint32_t kAccCols = BN <= 128 ? 128u : 256u, kCols = MB * kAccCols;      // tensor-memory columns
  constexpr int kWarpLoad = MB * kGemmEpiWarps, kWarpMma = kWarpLoad + 1;
  __shared__ __align__(8) uint64_t bars[2 * kGemmMaxStages + 2];
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_s;
  const uint32_t base = (smem_u32(gemm_smem) + 1023u) & ~1023u;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  struct Tile { int n0, m0, z, k_first, KB; };
  const unsigned n_tiles = tiles.x * tiles.y * tiles.z;
  auto tile_at = [&](unsigned t) {
    Tile c;
    c.n0 = (int)(t % tiles.x) * BN; c.m0 = (int)(t / tiles.x % tiles.y) * (128 * MB); c.z = (int)(t / (tiles.x * tiles.y));
    c.k_first = c.z * k_per; c.KB = (min(k_all - c.k_first, k_per) + 63) / 64;
    return c;
  };
  const uint32_t bar0 = smem_u32(bars);
  auto FULL = [&](int s) { return bar0 + 8u * (uint32_t)s; };
  auto EMPTY = [&](int s) { return bar0 + 8u * (uint32_t)(kGemmStages + s); };
  const uint32_t ACC = bar0 + 8u * (uint32_t)(2 * kGemmStages), FREE = ACC + 8u;   // accumulators complete; read out
  if (tid == 0) {
    for (int s = 0; s < kGemmStages; ++s) { mbar_init(FULL(s), 1); mbar_init(EMPTY(s), 1); }
    mbar_init(ACC, 1);
    mbar_init(FREE, MB * kGemmEpiWarps * 32);
    abort_s = 0;
    fence_mbar_init();
  }
  if (warp == kWarpMma) {
    tmem_alloc(smem_u32(&tmem_slot), kCols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;
  bool ok = true;
  constexpr uint32_t kOffB = MB * 16384u;
  if (warp == kWarpLoad) {
    if (lane == 0) {
      int it = 0;                                          // blocks of 64 k so far
      for (unsigned t = blockIdx.x; t < n_tiles && ok; t += gridDim.x) {
        const Tile c = tile_at(t);
        for (int kb = 0; kb < c.KB; ++kb, ++it) {
          const int s = it % kGemmStages;
          if (it >= kGemmStages && !gemm_wait(EMPTY(s), (uint32_t)((it / kGemmStages - 1) & 1))) { ok = false; break; }
          const uint32_t st = base + (uint32_t)s * kGemmStageBytes;
          mbar_expect_tx(FULL(s), kGemmStageBytes);
          const int kt = c.k_first + kb * 64;
          const int part = kt >= k_part ? kt >= 2 * k_part ? 2 : 1 : 0;
          const int k = kt - part * k_part;
          const CUtensorMap *ma = part == 2 ? &map_a3 : &map_a, *mb = part == 2 ? &map_b3 : part == 1 ? &map_b2 : &map_b;
          // K-major: one box of 64 k by all rows; MN-major: slabs of 64 columns by 64 k, 8 KB each
          if (AK) {
            tma_load_2d(st, ma, k, c.m0, FULL(s));
          } else {
#pragma unroll
            for (int i = 0; i < 2 * MB; ++i) tma_load_2d(st + i * 8192, ma, c.m0 + i * 64, k, FULL(s));
          }
          if (BK) {
            tma_load_2d(st + kOffB, mb, k, c.n0, FULL(s));
          } else {
#pragma unroll
            for (int i = 0; i < BN / 64; ++i) tma_load_2d(st + kOffB + i * 8192, mb, c.n0 + i * 64, k, FULL(s));
          }
        }
      }
    }
  } else if (warp == kWarpMma) {
    if (lane == 0) {
      const uint64_t desc_hi = smem_desc_sw128(0, 0) & 0xFFFFFFFF00000000ull;
      constexpr uint32_t idesc = idesc_bf16_f32(128, BN) | (AK ? 0u : 1u << 15) | (BK ? 0u : 1u << 16);   // bits: MN-major
      // MN-major: 64-column slabs 8192 bytes apart, 8-row groups (along k) 1024 bytes apart; 16 k are 2048 bytes.
      // K-major: 16 k are 32 bytes along the rows.
      constexpr uint32_t kSlab = (uint32_t)(8192 >> 4) << 16;
      constexpr uint32_t a_step = AK ? 2u : (2048u >> 4), b_step = BK ? 2u : (2048u >> 4);
      auto lo = [&](uint32_t at, bool kmajor) {
        return kmajor ? (uint32_t)(smem_desc_sw128(at, 0) & 0xFFFFFFFFull) : ((at & 0x3FFFFu) >> 4) | kSlab;
      };
      int it = 0;
      uint32_t done = 0;                                   // tiles issued
      for (unsigned t = blockIdx.x; t < n_tiles && ok; t += gridDim.x, ++done) {
        if (done > 0 && !gemm_wait(FREE, (done - 1) & 1u)) { ok = false; break; }
        tc_fence_after();
        const int KB = tile_at(t).KB;
        for (int kb = 0; kb < KB; ++kb, ++it) {
          const int s = it % kGemmStages;
          if (!gemm_wait(FULL(s), (uint32_t)((it / kGemmStages) & 1))) { ok = false; break; }
          tc_fence_after();
          const uint32_t st = base + (uint32_t)s * kGemmStageBytes;
          const uint32_t b_lo = lo(st + kOffB, BK);
#pragma unroll
          for (int kk = 0; kk < 4; ++kk)
#pragma unroll
            for (int mb = 0; mb < MB; ++mb)
              tc_mma_bf16(tmem + (uint32_t)mb * kAccCols, desc_hi | (lo(st + mb * 16384u, AK) + (uint32_t)kk * a_step),
                          desc_hi | (b_lo + (uint32_t)kk * b_step), idesc, (kb | kk) ? 1u : 0u);
          tc_commit(EMPTY(s));
        }
        tc_commit(ACC);
      }
    }
  }
  if (warp >= kWarpLoad) {          // a producer or issuer that gave up tells the epilogue not to wait for ever
    if (!ok && lane == 0) { abort_s = 1; atomicOr(flags, XKV_FLAG_TIMEOUT); }
  } else {
    // ---- epilogue: thread = accumulator lane = row m0 + tid
    uint32_t par = 0;
    for (unsigned t = blockIdx.x; t < n_tiles; t += gridDim.x, par ^= 1u) {
      const Tile c = tile_at(t);
      float* const Cz = Cf ? Cf + (size_t)c.z * M * ldc : nullptr;
      bool done = false;
      for (uint32_t i = 0; i < kGemmWaitLimit && !done; ++i) {
        done = mbar_try_wait(ACC, par);
        if (!done && (i & 1023u) == 1023u && *(volatile int*)&abort_s) break;
      }
      if (!done) {
        if (tid == 0) atomicOr(flags, XKV_FLAG_TIMEOUT);
        break;
      }
      tc_fence_after();
      const int m = c.m0 + tid;
      const uint32_t lane_base = ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(warp >> 2) * kAccCols;
      if (!Cf && c.n0 + BN <= N && (TRANS || (ldc & 7) == 0)) {
        // bf16 alone: to registers, the accumulators handed back, then the stores; as many columns at a time as registers
        // hold.  (Two parts of 192 columns spill 48 bytes at 96; 64 at a time spill nothing and hand the accumulators back
        // later: X Z in two parts, 131072 x 4096 x 576, 844 -> 849 us.)
        constexpr int kPart = BN == 192 ? 96 : LO ? 64 : 128;
#pragma unroll 1
        for (int n = 0; n < BN; n += kPart) {
          uint32_t h[kPart / 2], rest[LO ? kPart / 2 : 1];
#pragma unroll
          for (int cb = 0; cb < kPart / 32; ++cb) {
            float v[32];
            tmem_ld32(tmem + lane_base + (uint32_t)(n + cb * 32), v);
            tc_wait_ld();
#pragma unroll
            for (int i = 0; i < 16; ++i) {
              const __nv_bfloat162 two = __floats2bfloat162_rn(v[2 * i], v[2 * i + 1]);
              h[cb * 16 + i] = *reinterpret_cast<const uint32_t*>(&two);
              if (LO) {
                const __nv_bfloat162 out = __floats2bfloat162_rn(2.0f * (v[2 * i] - __low2float(two)), 2.0f * (v[2 * i + 1] - __high2float(two)));
                rest[cb * 16 + i] = *reinterpret_cast<const uint32_t*>(&out);
              }
            }
          }
          if (n + kPart == BN) {
            tc_fence_before();
            mbar_arrive(FREE);
          }
          if (m < M) {
            if (TRANS) {
              uint16_t* to = reinterpret_cast<uint16_t*>(Cb) + (long long)(c.n0 + n) * ldc + m;
              const long long to_rest = LO ? Cl - Cb : 0;
#pragma unroll
              for (int i = 0; i < kPart; ++i, to += ldc) {
                asm volatile("" : "+l"(to));               // one address at a time, not all of them in registers
                *to = (uint16_t)((i & 1) ? h[i >> 1] >> 16 : h[i >> 1]);
                if (LO) to[to_rest] = (uint16_t)((i & 1) ? rest[i >> 1] >> 16 : rest[i >> 1]);
              }
            } else {
              uint4* to = reinterpret_cast<uint4*>(Cb + (long long)m * ldc + c.n0 + n);
#pragma unroll
              for (int i = 0; i < kPart / 8; ++i) to[i] = make_uint4(h[4 * i], h[4 * i + 1], h[4 * i + 2], h[4 * i + 3]);
            }
          }
        }
      } else {
#pragma unroll 1
        for (int cb = 0; cb < BN / 32; ++cb) {
          float v[32];
          tmem_ld32(tmem + lane_base + (uint32_t)(cb * 32), v);
          tc_wait_ld();
          if (m < M) {
            const int nb = c.n0 + cb * 32;
            if (!TRANS && nb + 32 <= N && (ldc & 7) == 0) {
              // a whole run of 32 columns of one row: 16-byte stores (the row pitch keeps them aligned)
              const long long at = (long long)m * ldc + nb;
              if (Cz) {
#pragma unroll
                for (int i = 0; i < 32; i += 4) *reinterpret_cast<float4*>(Cz + at + i) = make_float4(v[i], v[i + 1], v[i + 2], v[i + 3]);
              }
              if (Cb) {
#pragma unroll
                for (int i = 0; i < 32; i += 8) {
                  __nv_bfloat162 h0 = __floats2bfloat162_rn(v[i], v[i + 1]), h1 = __floats2bfloat162_rn(v[i + 2], v[i + 3]);
                  __nv_bfloat162 h2 = __floats2bfloat162_rn(v[i + 4], v[i + 5]), h3 = __floats2bfloat162_rn(v[i + 6], v[i + 7]);
                  uint4 u;
                  u.x = *reinterpret_cast<uint32_t*>(&h0); u.y = *reinterpret_cast<uint32_t*>(&h1);
                  u.z = *reinterpret_cast<uint32_t*>(&h2); u.w = *reinterpret_cast<uint32_t*>(&h3);
                  *reinterpret_cast<uint4*>(Cb + at + i) = u;
                }
              }
            } else {
#pragma unroll
              for (int i = 0; i < 32; ++i) {
                const int n = nb + i;
                if (n < N) {
                  const long long at = TRANS ? (long long)n * ldc + m : (long long)m * ldc + n;
                  if (Cz) Cz[at] = v[i];
                  if (Cb) {
                    const __nv_bfloat16 hi = __float2bfloat16(v[i]);
                    Cb[at] = hi;
                    if (LO) Cl[at] = __float2bfloat16(2.0f * (v[i] - __bfloat162float(hi)));
                  }
                }
              }
            }
          }
        }
        tc_fence_before();
        mbar_arrive(FREE);
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == kWarpMma) {
    tc_fence_after();
    tmem_dealloc(tmem, kCols);
  }
}

}  // namespace

// ---------------------------------------------------------------------------------------------
// The small matrices (l x l, N x l).
namespace {

// ---- fp64 pieces of the Cholesky QR, on the fp64 tensor-core path (mma.sync m8n8k4) ----
constexpr int kDgemmLd = 68;                         // doubles per staged row of 64: 4 mod 16, so fragment loads are conflict free
__device__ __forceinline__ void dmma_8x8x4(double (&d)[2], double a, double b) {
  asm volatile("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0,%1}, {%2}, {%3}, {%0,%1};"
               : "+d"(d[0]), "+d"(d[1]) : "d"(a), "d"(b));
}

// Gram matrix U^T U of the fp32 iterate U (n x l), accumulated in fp64 because its condition number is the square of
// the iterate's: part[z][l][l] for the rows [z * rows_per, (z + 1) * rows_per), 64 x 64 tiles of the lower triangle.
// The rows are split so that the tiles fill the SMs about twice (81 full tiles of a 576 x 576 matrix, one CTA per SM
// and all 4096 rows each, took 193 us; half the tiles over six row ranges 61 us); the partial sums are added in a fixed
// order by the factorisation.  8 warps of 16 x 32, chunks of 32 rows widened to fp64 on their way into shared memory.
__global__ void __launch_bounds__(256)
gram_kernel(const float* __restrict__ U, double* __restrict__ part, int n, int l, int rows_per) {
  __shared__ double As[32][kDgemmLd], Bs[32][kDgemmLd];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int wm = (warp & 3) * 16, wn = (warp >> 2) * 32;
  int ti = 0, tj = blockIdx.x;                        // tile (ti, tj), tj <= ti
  while (tj > ti) { ++ti; tj -= ti; }
  const int m0 = ti * 64, n0 = tj * 64;
  const int k_begin = blockIdx.y * rows_per, k_end = min(n, k_begin + rows_per);
  const int lr = tid >> 4, lc = (tid & 15) * 4;       // this thread's piece of a staged chunk: rows lr, lr + 16; 4 columns
  double acc[2][4][2];
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) { acc[i][j][0] = 0.0; acc[i][j][1] = 0.0; }
  float4 pa[2], pb[2];
  auto fetch = [&](int k0) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int k = k0 + lr + 16 * h;
      const float4 z = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
      pa[h] = k < k_end ? *reinterpret_cast<const float4*>(U + (size_t)k * l + m0 + lc) : z;
      pb[h] = k < k_end ? *reinterpret_cast<const float4*>(U + (size_t)k * l + n0 + lc) : z;
    }
  };
  fetch(k_begin);
  for (int k0 = k_begin; k0 < k_end; k0 += 32) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      double* da = &As[lr + 16 * h][lc];
      double* db = &Bs[lr + 16 * h][lc];
      da[0] = (double)pa[h].x; da[1] = (double)pa[h].y; da[2] = (double)pa[h].z; da[3] = (double)pa[h].w;
      db[0] = (double)pb[h].x; db[1] = (double)pb[h].y; db[2] = (double)pb[h].z; db[3] = (double)pb[h].w;
    }
    __syncthreads();
    if (k0 + 32 < k_end) fetch(k0 + 32);              // the next chunk travels while this one is multiplied
#pragma unroll
    for (int kk = 0; kk < 32; kk += 4) {
      double a[2], b[4];
#pragma unroll
      for (int i = 0; i < 2; ++i) a[i] = As[kk + (lane & 3)][wm + 8 * i + (lane >> 2)];
#pragma unroll
      for (int j = 0; j < 4; ++j) b[j] = Bs[kk + (lane & 3)][wn + 8 * j + (lane >> 2)];
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) dmma_8x8x4(acc[i][j], a[i], b[j]);
    }
    __syncthreads();
  }
  double* C = part + (size_t)blockIdx.y * l * l;
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j)
      *reinterpret_cast<double2*>(C + (size_t)(m0 + wm + 8 * i + (lane >> 2)) * l + n0 + wn + 8 * j + 2 * (lane & 3)) =
          make_double2(acc[i][j][0], acc[i][j][1]);
}

// A grid-wide barrier of cooperative kernels: an arrival counter that only grows, polled by everybody (an arrival and
// one poll are the only trips to L2).  The wait is bounded like every wait of the library: a CTA that gives up raises
// XKV_FLAG_TIMEOUT and the abort word, and every other CTA leaves at its next wait.  Data that crosses it is read past
// L1 (other SMs wrote it).
constexpr unsigned kGridSpinLimit = 1u << 18;   // polls of a barrier that normally opens within microseconds
struct GridSync {            // words of the workspace's flag block
  unsigned int* flags;       // status word
  unsigned int* count;       // arrivals so far (monotonic)
  unsigned int* abort;       // a CTA gave up
  unsigned int spin_limit;   // polls of one barrier wait
  unsigned int no_arrival;   // fault injection (tests of the give-up path): CTA 0 arrives at no barrier, and passes the first
};
__device__ __forceinline__ unsigned ld_acquire_u32(const unsigned int* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void red_release_u32(unsigned int* p, unsigned v) {
  asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
// Returns false when the barrier was abandoned (by this CTA or another one).  `arrived` counts the arrivals expected so
// far: it starts at the counter's value before the kernel, the same in every CTA.
__device__ __forceinline__ bool grid_barrier(const GridSync& sy, unsigned& arrived, int* ok_s) {
  __syncthreads();
  const bool first = arrived == 0u;
  arrived += gridDim.x;
  if (threadIdx.x == 0) {
    const bool silent = sy.no_arrival != 0u && blockIdx.x == 0;
    bool ok = true;
    __threadfence();
    if (!silent) red_release_u32(sy.count, 1u);
    if (!silent || !first) {
      for (unsigned i = 0; ld_acquire_u32(sy.count) < arrived;) {
        if (++i >= sy.spin_limit || ((i & 15u) == 0u && ld_acquire_u32(sy.abort) != 0u)) { ok = false; break; }
      }
    }
    if (!ok) { atomicOr(sy.flags, XKV_FLAG_TIMEOUT); atomicExch(sy.abort, 1u); }
    __threadfence();
    *ok_s = ok ? 1 : 0;
  }
  __syncthreads();
  return *ok_s != 0;
}

// 1/sqrt(d) for d > 0 from the fp32 value y (relative error 2^-22): with e = 1 - d y^2 the binomial series y (1 - e)^-1/2 to
// its second order leaves 5/16 e^3, below the rounding.  (Four dependent operations; two steps of Newton's iteration are six.)
// The argument is scaled into [1, 4) by an even power of two first.
__device__ __forceinline__ double series_rsqrt(double d) {
  const int hi = __double2hiint(d);
  const int e = ((hi >> 20) - 1023) & ~1;                      // even exponent
  const double m = __hiloint2double(hi - (e << 20), __double2loint(d));
  double y = (double)rsqrtf((float)m);
  const double err = fma(-m * y, y, 1.0);
  y = fma(y * err, fma(0.375, err, 0.5), y);
  return __hiloint2double(__double2hiint(y) - ((e >> 1) << 20), __double2loint(y));
}

// Cholesky factorisation in fp64 of G + shift_rel * max_diag(G) * I and the inverse W = L^-1 of its factor, one
// cooperative kernel.  Blocks of 32.  At step p every lower tile (i, k), i >= p, is one item:
//   i > p, k > p    A_ik -= L_ip L_kp^T; the two blocks of the panel, L_ip = A_ip inv(L_pp)^T and L_kp, are formed by the item
//                   itself (they cost less than handing them over would); tile (p+1, p+1) is then factored at once, so that
//                   one grid barrier per step suffices
//   i > p, k <= p   the same elimination on the identity, R_ik -= L_ip W_pk (R starts as I), with W_pk = inv(L_pp) R_pk
//   i == p          W_pk is written
// A latency chain: 576 columns two by two in the diagonal blocks, 19 barriers.  (As three launches per panel the
// factorisation of a 576 x 576 matrix was 52 launches of 7 to 16 us; with the inverse formed after it, column by column, the
// kernel took 321 us, with the inverse carried along and a column a step 234, now 178.)  With W at hand the solve is a product.
// Buffers: part [n_part][l][l] partial Gram matrices (lower tiles of 64), Gm [l][l] the working matrix, Rt [l][l] the tiles
// of R below the diagonal, each transposed, Iv [l/32][32][32] inverses of the diagonal blocks, W [l][l] lower.
constexpr int kCholNb = 32, kCholThreads = 256, kCholLd = 36;   // 36 doubles per staged row: 4 mod 16, conflict free fragments

// One 8-row, 32-deep fragment product: acc (8 x 8 per tile) += A rows [m8..m8+7] of a staged block times B rows^T.
__device__ __forceinline__ void dmma_block(double (&acc)[2], const double* A, const double* B, int lane, double sign) {
#pragma unroll
  for (int kk = 0; kk < kCholNb; kk += 4)
    dmma_8x8x4(acc, sign * A[(lane >> 2) * kCholLd + kk + (lane & 3)], B[(lane >> 2) * kCholLd + kk + (lane & 3)]);
}

__global__ void __launch_bounds__(kCholThreads, 1)
chol_inverse_kernel(const double* __restrict__ part, int n_part, double* __restrict__ Gm, double* __restrict__ Rt,
                    double* __restrict__ Iv, double* __restrict__ W, int l, double shift_rel, unsigned arrived, GridSync sy) {
  __shared__ double A_s[kCholNb * kCholLd], B_s[kCholNb * kCholLd], V_s[kCholNb * kCholLd], Li_s[kCholNb * kCholLd], Lk_s[kCholNb * kCholLd];
  __shared__ double red_s[kCholThreads / 32];
  __shared__ int ok_s;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nb = gridDim.x, bid = blockIdx.x;
  const int nbk = l / kCholNb;
  // ---- the Gram matrix: partial sums added in order, every CTA a share of the elements of the lower 64 x 64 tiles
  for (long long e2 = (long long)bid * kCholThreads + tid; e2 < (long long)l * l / 2; e2 += (long long)nb * kCholThreads) {
    const int row = (int)(e2 / (l / 2)), c = (int)(e2 % (l / 2)) * 2;
    if (c / 64 > row / 64) continue;
    double2 v = make_double2(0.0, 0.0);
    for (int z = 0; z < n_part; ++z) {
      const double2 u = *reinterpret_cast<const double2*>(part + ((size_t)z * l + row) * l + c);
      v.x += u.x; v.y += u.y;
    }
    *reinterpret_cast<double2*>(Gm + (size_t)row * l + c) = v;
  }
  if (!grid_barrier(sy, arrived, &ok_s)) return;
  double shift;
  {
    double mx = 0.0;
    for (int i = tid; i < l; i += kCholThreads) mx = fmax(mx, __ldcg(Gm + (size_t)i * l + i));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if (lane == 0) red_s[warp] = mx;
    __syncthreads();
    mx = red_s[lane & (kCholThreads / 32 - 1)];
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    shift = shift_rel * mx;
  }
  auto stage = [&](double* dst, const double* src, int ld) {   // a 32 x 32 block
    for (int e = tid; e < kCholNb * kCholNb / 2; e += kCholThreads) {
      const int r = e >> 4, c = (e & 15) * 2;
      const double2 v = __ldcg(reinterpret_cast<const double2*>(src + (size_t)r * ld + c));
      dst[r * kCholLd + c] = v.x; dst[r * kCholLd + c + 1] = v.y;
    }
  };
  const int t_m = warp & 3, t_n = (warp >> 2) * 2;             // this warp's 8 x 8 tiles of a 32 x 32 block: (t_m, t_n), (t_m, t_n + 1)
  auto put = [&](double* dst, int ld, const double (&acc)[2][2]) {
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      double* d = dst + (size_t)(t_m * 8 + (lane >> 2)) * ld + (t_n + j) * 8 + 2 * (lane & 3);
      d[0] = acc[j][0]; d[1] = acc[j][1];
    }
  };
  // ---- factor the diagonal block in A_s and invert the factor, two columns a step, which halves the chain of reciprocal
  // roots: with the pivots a, b, d the second root is that of a d - b^2 and does not wait for the first.  Warps 0-3 hold the
  // matrix, lane = row, warps 4-7 the inverse, lane = column; the pair of columns (of rows, in the inverse) 2 s, 2 s + 1
  // belongs to warp s mod 4 of either.  A step is one barrier: the owner brings its pair up to date, works the columns out
  // and hands them over; the others then take them off their pairs, the owner of the next step after its own barrier.  The
  // inverse is one step behind.  A pivot that is not positive (breakdown) is replaced by a tiny one and reported.
  auto factor = [&](int p) {
    __syncthreads();
    double* const col = B_s;                                   // [step & 3][2][32] columns of the factor
    double* const row = B_s + 4 * 2 * kCholNb;                 // [step & 3][2][32] rows of the inverse
    double* const piv = row + 4 * 2 * kCholNb;                 // [step & 3][3] 1 / l_11, l_21, 1 / l_22
    const bool inverse = warp >= 4;
    const int own = warp & 3;
    double a[4][2];
#pragma unroll
    for (int k = 0; k < 4; ++k)
#pragma unroll
      for (int x = 0; x < 2; ++x) {
        const int j = 2 * (4 * k + own) + x;
        a[k][x] = inverse ? (j == lane ? 1.0 : 0.0) : A_s[lane * kCholLd + j];
      }
    auto take_off = [&](double (&v)[2], int of, int step) {    // step's columns (and rows) off pair `of`
      const double* const c = col + (step & 3) * 2 * kCholNb + 2 * of;
      const double* const m = (inverse ? row : col) + (step & 3) * 2 * kCholNb + lane;
      const double m0 = m[0], m1 = m[kCholNb];
#pragma unroll
      for (int x = 0; x < 2; ++x) v[x] = fma(-m1, c[kCholNb + x], fma(-m0, c[x], v[x]));
    };
#pragma unroll
    for (int k = 0; k < 4; ++k) {
#pragma unroll 1
      for (int w = 0; w < 4; ++w) {
        const int st = 4 * k + w;
        double* const my_piv = piv + (st & 3) * 3;
        if (!inverse && own == w) {
          if (st > 0) take_off(a[k], st, st - 1);
          double a0 = __shfl_sync(0xffffffffu, a[k][0], 2 * st);
          const double b0 = __shfl_sync(0xffffffffu, a[k][0], 2 * st + 1), d0 = __shfl_sync(0xffffffffu, a[k][1], 2 * st + 1);
          const bool bad_a = !(a0 > 0.0);
          a0 = bad_a ? 1e-300 : a0;
          const double det = fma(a0, d0, -(b0 * b0));
          const bool bad_d = !(det > 0.0);
          const double y1 = series_rsqrt(a0), y2 = series_rsqrt(bad_d ? 1.0 : det);
          const double l21 = b0 * y1, i22 = bad_d ? 1e150 : y2 * (a0 * y1), l22 = bad_d ? 1e-150 : det * y2 * y1;
          const double x1 = (lane == 2 * st ? a0 : a[k][0]) * y1;
          const double x2 = lane == 2 * st + 1 ? l22 : fma(-x1, l21, a[k][1]) * i22;
          double* const c = col + (st & 3) * 2 * kCholNb + lane;
          c[0] = x1; c[kCholNb] = x2;
          if (lane == 0) {
            my_piv[0] = y1; my_piv[1] = l21; my_piv[2] = i22;
            if (bad_a || bad_d) atomicOr(sy.flags, XKV_FLAG_CLF_BREAKDOWN);
          }
        }
        named_bar_sync(1, kCholThreads);
        if (inverse) {
          if (st > 0) {
#pragma unroll
            for (int j = k; j < 4; ++j)
              if (j > k || own >= w) take_off(a[j], 4 * j + own, st - 1);
          }
          if (own == w) {
            a[k][0] *= my_piv[0];
            a[k][1] = fma(-my_piv[1], a[k][0], a[k][1]) * my_piv[2];
            double* const c = row + (st & 3) * 2 * kCholNb + lane;
            c[0] = a[k][0]; c[kCholNb] = a[k][1];
#pragma unroll
            for (int x = 0; x < 2; ++x) Iv[((size_t)p * kCholNb + 2 * st + x) * kCholNb + lane] = 2 * st + x >= lane ? a[k][x] : 0.0;
          }
        } else if (own != ((w + 1) & 3)) {
#pragma unroll
          for (int j = k; j < 4; ++j)
            if (j > k || own > w) {
              if (own == w && st > 0) take_off(a[j], 4 * j + own, st - 1);
              take_off(a[j], 4 * j + own, st);
            }
        }
      }
    }
  };
  auto first_of = [&](int i) { return i * (i + 1) / 2; };      // tiles of the lower triangle, row by row
  auto tile_of = [&](int t, int& i, int& k) { i = 0; k = t; while (k > i) { ++i; k -= i; } };
  if (bid == 0) {
    stage(A_s, Gm, l);
    __syncthreads();
    if (tid < kCholNb) A_s[tid * kCholLd + tid] += shift;
    factor(0);
  }
  if (!grid_barrier(sy, arrived, &ok_s)) return;
  const int fr = t_m * 8 + (lane >> 2), fc = 2 * (lane & 3);   // this thread's fragment: row fr, columns (t_n + j) * 8 + fc, + 1
  for (int p = 0; p < nbk; ++p) {
    // CTA 0 takes the tile whose factor everybody waits for, the others share the rest
    const int critical = p + 1 < nbk ? first_of(p + 1) + p + 1 : -1, items = first_of(nbk) - first_of(p) - (critical >= 0 ? 1 : 0);
    for (int e = bid == 0 ? items : bid - 1;; e += nb - 1) {
      const bool crit = bid == 0 && critical >= 0;
      if (!crit && e >= items) break;
      int t = crit ? critical : first_of(p) + e;
      if (!crit && critical >= 0 && t >= critical) ++t;
      int i, k;
      tile_of(t, i, k);
      const bool trail = k > p;
      __syncthreads();
      stage(V_s, Iv + (size_t)p * kCholNb * kCholNb, kCholNb);
      if (i > p) stage(A_s, Gm + (size_t)i * kCholNb * l + p * kCholNb, l);
      if (trail ? i != k : k < p) stage(B_s, (trail ? Gm + (size_t)k * kCholNb * l + p * kCholNb : Rt + (size_t)p * kCholNb * l + k * kCholNb), l);
      double acc[2][2] = {{0.0, 0.0}, {0.0, 0.0}};
      double* const own = (trail ? Gm : Rt) + (size_t)i * kCholNb * l + k * kCholNb;
      if (i > p && (trail || k < p)) {
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          const double2 v = __ldcg(reinterpret_cast<const double2*>(own + (size_t)fr * l + (t_n + j) * 8 + fc));
          acc[j][0] = v.x; acc[j][1] = v.y;
        }
      }
      __syncthreads();
      double li[2][2] = {{0.0, 0.0}, {0.0, 0.0}}, lk[2][2] = {{0.0, 0.0}, {0.0, 0.0}};
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        if (i > p) dmma_block(li[j], A_s + t_m * 8 * kCholLd, V_s + (t_n + j) * 8 * kCholLd, lane, 1.0);
        // L_kp, or W_pk^T = R_pk^T inv(L_pp)^T
        if (trail ? i != k : k < p) dmma_block(lk[j], B_s + t_m * 8 * kCholLd, V_s + (t_n + j) * 8 * kCholLd, lane, 1.0);
        else if (!trail) { lk[j][0] = V_s[((t_n + j) * 8 + fc) * kCholLd + fr]; lk[j][1] = V_s[((t_n + j) * 8 + fc + 1) * kCholLd + fr]; }
      }
      if (i == p) {
#pragma unroll
        for (int j = 0; j < 2; ++j)
#pragma unroll
          for (int x = 0; x < 2; ++x) W[(size_t)(p * kCholNb + (t_n + j) * 8 + fc + x) * l + k * kCholNb + fr] = lk[j][x];
        continue;
      }
      put(Li_s, kCholLd, li);
      if (i != k) put(Lk_s, kCholLd, lk);
      __syncthreads();
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        if (trail) {
          if (i == k && p == 0) {                              // first touch of a diagonal tile
#pragma unroll
            for (int x = 0; x < 2; ++x) if (fr == (t_n + j) * 8 + fc + x) acc[j][x] += shift;
          }
          dmma_block(acc[j], Li_s + t_m * 8 * kCholLd, (i != k ? Lk_s : Li_s) + (t_n + j) * 8 * kCholLd, lane, -1.0);
        } else {
          dmma_block(acc[j], Lk_s + t_m * 8 * kCholLd, Li_s + (t_n + j) * 8 * kCholLd, lane, -1.0);
        }
      }
      if (crit) {
        put(A_s, kCholLd, acc);
        factor(p + 1);
        break;
      }
      put(own, l, acc);
    }
    if (p + 1 < nbk && !grid_barrier(sy, arrived, &ok_s)) return;
  }
}

// Z (n x l) = U W^T for the lower-triangular W = L^-1 (fp64): 64 x 64 tiles, tile column J takes the first J + 1 blocks of
// 64.  Longest tiles first.  Also writes the bf16 copy the tensor-core products read, and behind it (n rows on) the bf16 of
// what the copy leaves out.  (The blocked triangular solve that
// kept 32 rows of Z in shared memory took 161 us and 69 us for the inverses of its diagonal blocks at 4096 x 576; this
// product 59 us.)
__global__ void __launch_bounds__(256)
tri_product_kernel(const float* __restrict__ U, const double* __restrict__ W, float* __restrict__ Z,
                   __nv_bfloat16* __restrict__ Zb, int n, int l) {
  __shared__ double As[64][kCholLd], Bs[64][kCholLd];          // 32 k of 64 rows of U, of 64 rows of W
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int wm = (warp & 3) * 16, wn = (warp >> 2) * 32;
  const int J = l / 64 - 1 - blockIdx.y, row0 = blockIdx.x * 64, n0 = J * 64;
  const int k_end = (J + 1) * 64;
  double acc[2][4][2];
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) { acc[i][j][0] = 0.0; acc[i][j][1] = 0.0; }
  float4 pa[2];
  double2 pb[4];
  const int ar = tid >> 3, ac = (tid & 7) * 4;                 // U: rows ar, ar + 32; 4 columns
  const int br = tid >> 4, bc = (tid & 15) * 2;                // W: rows br + 16 h; 2 columns
  auto fetch = [&](int k0) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int r = row0 + ar + 32 * h;
      pa[h] = r < n ? *reinterpret_cast<const float4*>(U + (size_t)r * l + k0 + ac) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    }
#pragma unroll
    for (int h = 0; h < 4; ++h) {
      const int j = n0 + br + 16 * h, k = k0 + bc;             // above the diagonal W is not stored
      pb[h] = make_double2(0.0, 0.0);
      if (k / kCholNb <= j / kCholNb) pb[h] = *reinterpret_cast<const double2*>(W + (size_t)j * l + k);
    }
  };
  fetch(0);
  for (int k0 = 0; k0 < k_end; k0 += 32) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      double* d = &As[ar + 32 * h][ac];
      d[0] = (double)pa[h].x; d[1] = (double)pa[h].y; d[2] = (double)pa[h].z; d[3] = (double)pa[h].w;
    }
#pragma unroll
    for (int h = 0; h < 4; ++h) { Bs[br + 16 * h][bc] = pb[h].x; Bs[br + 16 * h][bc + 1] = pb[h].y; }
    __syncthreads();
    if (k0 + 32 < k_end) fetch(k0 + 32);
#pragma unroll
    for (int kk = 0; kk < 32; kk += 4) {
      double a[2], b[4];
#pragma unroll
      for (int i = 0; i < 2; ++i) a[i] = As[wm + 8 * i + (lane >> 2)][kk + (lane & 3)];
#pragma unroll
      for (int j = 0; j < 4; ++j) b[j] = Bs[wn + 8 * j + (lane >> 2)][kk + (lane & 3)];
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) dmma_8x8x4(acc[i][j], a[i], b[j]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int r = row0 + wm + 8 * i + (lane >> 2), c = n0 + wn + 8 * j + 2 * (lane & 3);
      if (r < n) {
        const float z0 = (float)acc[i][j][0], z1 = (float)acc[i][j][1];
        *reinterpret_cast<float2*>(Z + (size_t)r * l + c) = make_float2(z0, z1);
        const __nv_bfloat162 hi = __floats2bfloat162_rn(z0, z1);
        const float2 h = __bfloat1622float2(hi);
        *reinterpret_cast<__nv_bfloat162*>(Zb + (size_t)r * l + c) = hi;
        *reinterpret_cast<__nv_bfloat162*>(Zb + (size_t)(n + r) * l + c) = __floats2bfloat162_rn(z0 - h.x, z1 - h.y);
      }
    }
}

}  // namespace

namespace {

// Eigen-decomposition of the symmetric l x l matrix M by block Jacobi in one cooperative kernel.  Blocks of 32 indices
// meet in round-robin (tournament) order: l/32 - 1 rounds per sweep, l/64 disjoint block pairs in a round.  A round:
//   A  one CTA per pair takes the pair's 64 x 64 submatrix through 32 rounds of 32 disjoint rotations between the two
//      blocks (in the first round of a sweep also once through the pairs inside each block) and publishes their product
//      Q; meanwhile the other CTAs bring the eigenvectors up to date with the Q of the round before;
//   B  the grid applies M <- Q^T M Q, 64 x 32 pieces, from one buffer to the other.
// Two grid barriers per 32 rounds of rotations.  (Applying every round of l/2 rotations to the whole matrix takes a
// barrier per round: 575 per sweep of a 576 x 576 matrix, 4.9 us each, 8.5 ms for three sweeps; taking the 64 x 64
// problems to convergence before they are applied was slower still.  This form took 1.5 ms for
// the same three sweeps and takes 1.22 with the cross rounds in registers.)  A check per sweep ends the sweeps once the
// off-diagonal weight is below kJacobiTol.  On return the eigenvalues are on the diagonal of M (buffer 0), the
// eigenvectors the rows of Pt.
constexpr int kJacobiMaxPairs = 1024;              // l <= 2048
constexpr int kJacobiSweeps = 16;
// The sweeps end when the off-diagonal weight (sum of squares) is below this fraction of the total.  The
// eigenvectors are stored as bf16 (relative rounding 2^-9); an off-diagonal residue of 1e-4 in relative norm is
// twenty times below that, and the convergence is quadratic.
constexpr float kJacobiTol = 1e-8f;
// And when the entries are small beside their own diagonal too: m_ij / sqrt(m_ii m_jj), rms, below this.  Where one
// direction holds nearly everything (an outlier row or column), the first condition holds before the first sweep, and the r
// largest of l diagonal entries are then not the r best directions: residual of a 3000 x 256 cache with one row a thousand
// times the others, rank 64, 1.049 x the optimum with no sweep, 1.024 with one, 1.018 with two, 1.017 converged.  Caches
// with a decaying spectrum are below it after one or two of their three to eight sweeps.  Diagonal entries below
// kJacobiFloor of the largest one, what the two-part Z and W leave of a direction that X does not have, count as that.
constexpr float kJacobiScaledTol = 5e-3f;
constexpr float kJacobiFloor = 1e-10f;
constexpr int kJacobiThreads = 1024;
constexpr int kJb = 32, kJp = 2 * kJb;             // indices of a block, of a pair
constexpr int kJacobiSmem = 4 * (kJp * kJp * 3 + 8 * kJp * kJb + kJp * (kJb + 1));   // bytes, see the carve-up
// Pair k of round t of the round-robin tournament of n (even) players, the smaller first.
__device__ __forceinline__ int2 tournament_pair(int k, int t, int n) {
  int p, q;
  if (k == 0) { p = n - 1; q = t; }
  else {
    p = t + k; if (p >= n - 1) p -= n - 1;
    q = t - k; if (q < 0) q += n - 1;
  }
  return p < q ? make_int2(p, q) : make_int2(q, p);
}

// The rotation (c, s) that annihilates a_pq: columns (p, q) become (c p - s q, s p + c q).  The formula is on the chain of
// every round (a cross round with all of the submatrix in shared memory: 1165 cycles, 918 with the formula left out), so each step is one approximate instruction and
// there is no branch.  |tau| too large to square gives t = 0 and the identity; so does an a_pq next to nothing.
// An error of t leaves a little of a_pq to the next sweep; an error of c^2 + s^2 stays, and thousands of rotations add theirs
// up, so the root takes a step of Newton's iteration.  Largest entry of P P^T - I, l = 576, 8 sweeps: 3.0e-4 without the
// step, 1.0e-4 with it (rotating one round at a time with IEEE divisions: 3.0e-4).
__device__ __forceinline__ float2 jacobi_rotation(float app, float aqq, float apq) {
  auto rcp = [](float x) { float y; asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x)); return y; };
  const float tau = (aqq - app) * rcp(2.0f * apq);
  float h, c;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(h) : "f"(fmaf(tau, tau, 1.0f)));
  const float t = copysignf(rcp(fabsf(tau) + h), tau);
  const float w = fmaf(t, t, 1.0f);                          // 1 .. 2
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(c) : "f"(w));
  c = fmaf(0.5f * c, fmaf(-w * c, c, 1.0f), c);
  return fabsf(apq) > 1e-30f ? make_float2(c, t * c) : make_float2(1.0f, 0.0f);
}

// out[r][c] = sum_k A[k][r] B[k][c] for A [64][64], B [64][ldb] in shared memory, 64 x 32 outputs, by 1024 threads:
// eight groups of eight k, 4 x 4 outputs per thread, partial sums through `red` [8][64][32].  The caller reads the sums
// with piece_sum after the barrier that ends this function.
__device__ __forceinline__ void piece_product(const float* __restrict__ A, const float* __restrict__ B, int ldb, float* __restrict__ red) {
  const int tid = threadIdx.x, grp = tid >> 7, e = tid & 127;
  const int r0 = (e >> 3) * 4, c0 = (e & 7) * 4;
  float acc[4][4] = {};
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int k = grp * 8 + i;
    const float4 av = *reinterpret_cast<const float4*>(A + k * kJp + r0), bv = *reinterpret_cast<const float4*>(B + k * ldb + c0);
    const float a[4] = {av.x, av.y, av.z, av.w}, b[4] = {bv.x, bv.y, bv.z, bv.w};
#pragma unroll
    for (int y = 0; y < 4; ++y)
#pragma unroll
      for (int x = 0; x < 4; ++x) acc[y][x] = fmaf(a[y], b[x], acc[y][x]);
  }
#pragma unroll
  for (int y = 0; y < 4; ++y)
    *reinterpret_cast<float4*>(red + grp * (kJp * kJb) + (r0 + y) * kJb + c0) = make_float4(acc[y][0], acc[y][1], acc[y][2], acc[y][3]);
  __syncthreads();
}
__device__ __forceinline__ float piece_sum(const float* __restrict__ red, int o) {
  float v = 0.0f;
#pragma unroll
  for (int g = 0; g < 8; ++g) v += red[g * (kJp * kJb) + o];
  return v;
}

// The 32 rounds of rotations (i, 32 + (i + t) mod 32) of a pair's 64 x 64 submatrix, in registers.  The matrix is symmetric:
// kept are its 2 x 2 blocks (a, a + e mod 32), e = 0 .. 16, that is rows a and a' = 32 + (a + t) mod 32 by columns b and b'
// of b = a + e.  Lane = a; warp w of the first four holds e = 4 w + 1 .. 4 w + 4, warp 0 e = 0 as well.  From round to round
// a' and b' move one on, so x01 comes from block e + 1 of the same lane, x10 from block e - 1 and x11 from block e of the
// next lane (across two warps through shared memory).  Warp 0 works the next round's rotations out of its blocks 0 and 1
// while the others still update theirs: the chain of a round is two rotations, the formula and one barrier.  Warps 4-11 hold
// Q, eight rows each, lane = columns i and 32 + (i + t) mod 32.
// (The full submatrix in shared memory, 16 warps and all of them computing the formula: 1165 cycles a round; the same in
// registers: 973.)
// A function of its own: it wants the registers that the rest of the kernel would keep.  Called by warps 0-11.
// X, Q0 [64][64]: submatrix and product so far; buf: room for 2 x 64 + 2 x 4 x 64 floats; Qout [64][64].
constexpr int kCrossWarps = 12;
__device__ __noinline__ void cross_rotations(const float* __restrict__ X, float* __restrict__ buf, const float* __restrict__ Q0,
                                             float* __restrict__ Qout) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, up = (lane + 1) & 31;
  float2* const cs_s = reinterpret_cast<float2*>(buf);       // [2][32]
  float* const ex_s = buf + 128;                             // [2][4]: x01 of a warp's first block, x10 of its last
  if (warp >= 4) {
    float qu[8], qv[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const float* row = Q0 + ((warp - 4) * 8 + k) * kJp;
      qu[k] = row[lane];
      qv[k] = row[kJb + lane];
    }
#pragma unroll 1
    for (int t = 0; t < kJb; ++t) {
      ptx::named_bar_sync(1, kCrossWarps * 32);
      const float2 cs = cs_s[(t & 1) * 32 + lane];
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const float u = qu[k], v = qv[k];
        qu[k] = cs.x * u - cs.y * v;
        qv[k] = __shfl_sync(0xffffffffu, cs.y * u + cs.x * v, up);
      }
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) {                            // after 32 moves the columns are back where they began
      float* row = Qout + ((warp - 4) * 8 + k) * kJp;
      row[lane] = qu[k];
      row[kJb + lane] = qv[k];
    }
    return;
  }
  float x00[5], x01[5], x10[5], x11[5];                      // block e = 4 warp + i (i = 0: warp 0 only)
#pragma unroll
  for (int i = 0; i < 5; ++i) {
    const int c = (lane + 4 * warp + i) & 31;
    x00[i] = X[lane * kJp + c]; x01[i] = X[lane * kJp + kJb + c];
    x10[i] = X[(kJb + lane) * kJp + c]; x11[i] = X[(kJb + lane) * kJp + kJb + c];
  }
  float2 cs = make_float2(1.0f, 0.0f);
  if (warp == 0) cs_s[lane] = cs = jacobi_rotation(x00[0], x11[0], x01[0]);
  // block i <- R_a^T block R_b for the rotations (ca, sa) of its rows, (cb, sb) of its columns
  auto turn = [&](int i, float ca, float sa, float cb, float sb) {
    const float u00 = cb * x00[i] - sb * x01[i], u01 = sb * x00[i] + cb * x01[i];
    const float u10 = cb * x10[i] - sb * x11[i], u11 = sb * x10[i] + cb * x11[i];
    x00[i] = ca * u00 - sa * u10; x01[i] = ca * u01 - sa * u11;
    x10[i] = sa * u00 + ca * u10; x11[i] = sa * u01 + ca * u11;
  };
#pragma unroll 1
  for (int t = 0; t < kJb; ++t) {
    ptx::named_bar_sync(1, kCrossWarps * 32);                // this round's rotations, the neighbours' blocks of the last
    float* const ex = ex_s + (t & 1) * 256;
    const float* const ex_last = ex_s + ((t + 1) & 1) * 256;
    if (warp != 0) {
      cs = cs_s[(t & 1) * 32 + lane];
      if (t > 0) x10[1] = ex_last[(warp - 1) * 64 + 32 + up];
    }
    if (t > 0 && warp < 3) x01[4] = ex_last[(warp + 1) * 64 + lane];
    const float ca = cs.x, sa = cs.y;
    auto turn_at = [&](int i) {
      const int from = (lane + 4 * warp + i) & 31;
      turn(i, ca, sa, __shfl_sync(0xffffffffu, ca, from), __shfl_sync(0xffffffffu, sa, from));
    };
    turn_at(1);
    if (warp == 0) {
      turn(0, ca, sa, ca, sa);
      x11[0] = __shfl_sync(0xffffffffu, x11[0], up);
      cs = jacobi_rotation(x00[0], x11[0], x01[1]);
      cs_s[((t + 1) & 1) * 32 + lane] = cs;
    }
#pragma unroll
    for (int i = 2; i < 5; ++i) turn_at(i);
    ex[warp * 64 + lane] = x01[1];
    ex[warp * 64 + 32 + lane] = x10[4];
    const float wrap = __shfl_sync(0xffffffffu, x10[3], (lane + 17) & 31);   // block (a, a + 17) is that of (a + 17, a), transposed
#pragma unroll
    for (int i = 4; i >= 2; --i) x10[i] = __shfl_sync(0xffffffffu, x10[i - 1], up);
    if (warp == 0) x10[1] = __shfl_sync(0xffffffffu, x10[0], up);
#pragma unroll
    for (int i = 0; i < 4; ++i) x01[i] = x01[i + 1];
    if (warp == 3) x01[4] = wrap;
    x10[0] = x01[0];
#pragma unroll
    for (int i = 1; i < 5; ++i) x11[i] = __shfl_sync(0xffffffffu, x11[i], up);
  }
}

__global__ void __launch_bounds__(kJacobiThreads, 1)
jacobi_block_kernel(float* __restrict__ M0, float* __restrict__ M1, float* __restrict__ Pt, float* __restrict__ Qg, int l,
                    float4* __restrict__ partial, unsigned arrived, GridSync sy) {
  extern __shared__ __align__(16) float js[];
  __shared__ int ok_s, done_s;
  __shared__ float3 red_s[kJacobiThreads / 32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nb = gridDim.x, bid = blockIdx.x;
  const int nblk = l / kJb, npair = l / kJp;                 // l is a multiple of 64
  const long long gtid = (long long)bid * kJacobiThreads + tid, gstride = (long long)nb * kJacobiThreads;
  for (long long e = gtid; e < (long long)l * l; e += gstride) Pt[e] = (e / l == e % l) ? 1.0f : 0.0f;
  float* const S0 = js;                                      // [64][64] each; phase A: the submatrix and its other buffer
  float* const S1 = S0 + kJp * kJp;
  float* const S2 = S1 + kJp * kJp;                          // phase A: the product of the rotations, Q
  float* const R = S2 + kJp * kJp;                           // [8][64][32] partial products; phase A: rotations of all rounds
  float* const T = R + 8 * kJp * kJb;                        // [64][33]
  float2* const cs_s = reinterpret_cast<float2*>(R);         // [63][32]
  // position i of pair pq (0..63) in the whole matrix
  auto at = [&](int2 pq, int i) { return (i < kJb ? pq.x : pq.y) * kJb + (i & (kJb - 1)); };

  // ---- A: rotations of one pair
  auto solve_pair = [&](const float* M, int2 pq, bool inside, float* Qout) {
    __syncthreads();
    for (int e = tid; e < kJp * kJp; e += kJacobiThreads) {
      S0[e] = __ldcg(M + (size_t)at(pq, e >> 6) * l + at(pq, e & 63));
      S2[e] = (e >> 6) == (e & 63) ? 1.0f : 0.0f;
    }
    __syncthreads();
    float* X = S0;
    float* Xn = S1;
    // one round of 32 disjoint rotations: lane b of every warp works out rotation b (index pair (i, j)); warps 0-15
    // update the 2 x 2 blocks (a, b) of the submatrix for two a each
    auto round = [&](int i, int j, int slot, auto&& row) {   // row(a): index pair of rotation a
      const float2 cs = jacobi_rotation(X[i * kJp + i], X[j * kJp + j], X[i * kJp + j]);
      if (warp == 0) cs_s[slot * 32 + lane] = cs;
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const int a = warp * 2 + k;
        const int2 ij = row(a);
        const int ia = ij.x, ja = ij.y;
        const float ca = __shfl_sync(0xffffffffu, cs.x, a), sa = __shfl_sync(0xffffffffu, cs.y, a);
        const float x00 = X[ia * kJp + i], x01 = X[ia * kJp + j], x10 = X[ja * kJp + i], x11 = X[ja * kJp + j];
        const float u00 = cs.x * x00 - cs.y * x01, u01 = cs.y * x00 + cs.x * x01;
        const float u10 = cs.x * x10 - cs.y * x11, u11 = cs.y * x10 + cs.x * x11;
        Xn[ia * kJp + i] = ca * u00 - sa * u10; Xn[ia * kJp + j] = ca * u01 - sa * u11;
        Xn[ja * kJp + i] = sa * u00 + ca * u10; Xn[ja * kJp + j] = sa * u01 + ca * u11;
      }
    };
    if (inside) {
      // the pairs inside the two blocks: 31 rounds, lanes 0-15 in the first block, lanes 16-31 in the second
      for (int t = 0; t < kJb - 1; ++t) {
        const int2 ij = tournament_pair(lane & 15, t, kJb);
        const int off = (lane >> 4) * kJb;
        if (warp < 16)
          round(ij.x + off, ij.y + off, t, [&](int a) {
            return make_int2(__shfl_sync(0xffffffffu, ij.x + off, a), __shfl_sync(0xffffffffu, ij.y + off, a));
          });
        __syncthreads();
        float* x = X; X = Xn; Xn = x;
        if (warp >= 16) {                                    // (nobody writes this slot of cs_s again before the next barrier)
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            float* row = S2 + ((warp - 16) * 4 + k) * kJp + off;
            const float2 cs = cs_s[t * 32 + lane];
            const float u = row[ij.x], v = row[ij.y];
            row[ij.x] = cs.x * u - cs.y * v;
            row[ij.y] = cs.y * u + cs.x * v;
          }
        }
      }
    }
    __syncthreads();
    if (warp < kCrossWarps) cross_rotations(X, X == S0 ? S1 : S0, S2, Qout);   // (the other buffer is free)
  };
  // ---- eigenvectors: rows of pair pq, columns c0 .. c0 + 63 of Pt  <-  Q^T times them
  auto rotate_vectors = [&](int2 pq, int c0, const float* Q) {
    __syncthreads();
    for (int e = tid; e < kJp * kJp; e += kJacobiThreads) {
      S0[e] = __ldcg(Pt + (size_t)at(pq, e >> 6) * l + c0 + (e & 63));      // [k][column of Pt]
      S1[e] = __ldcg(Q + e);                                               // [k][new row]
    }
    __syncthreads();
#pragma unroll 1
    for (int h = 0; h < 2; ++h) {
      piece_product(S0, S1 + h * kJb, kJp, R);               // [column][new row of block h]
      for (int o = tid; o < kJp * kJb; o += kJacobiThreads) T[(o >> 5) * (kJb + 1) + (o & 31)] = piece_sum(R, o);
      __syncthreads();
      for (int o = tid; o < kJp * kJb; o += kJacobiThreads)
        Pt[(size_t)at(pq, h * kJb + (o >> 6)) * l + c0 + (o & 63)] = T[(o & 63) * (kJb + 1) + (o >> 6)];
      __syncthreads();
    }
  };
  // ---- B: one 64 x 32 piece of Q_a^T M Q_b (block h of pair b), and its mirror image
  auto rotate_matrix = [&](const float* M, float* Mn, int a, int b, int h, int t, const float* Q) {
    const int2 pa = tournament_pair(a, t, nblk), pb = tournament_pair(b, t, nblk);
    __syncthreads();
    for (int e = tid; e < kJp * kJp; e += kJacobiThreads) {
      S0[e] = __ldcg(M + (size_t)at(pb, e >> 6) * l + at(pa, e & 63));      // M is symmetric: [k in b][row in a]
      S1[e] = __ldcg(Q + (size_t)b * kJp * kJp + e);                       // [k in b][column]
      S2[e] = __ldcg(Q + (size_t)a * kJp * kJp + e);                       // [k in a][row]
    }
    __syncthreads();
    piece_product(S0, S1 + h * kJb, kJp, R);
    float v[2];
#pragma unroll
    for (int i = 0; i < 2; ++i) v[i] = piece_sum(R, tid + i * kJacobiThreads);
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 2; ++i) S0[tid + i * kJacobiThreads] = v[i];        // [k in a][column]
    __syncthreads();
    piece_product(S2, S0, kJb, R);
    for (int o = tid; o < kJp * kJb; o += kJacobiThreads) {
      const float y = piece_sum(R, o);
      Mn[(size_t)at(pa, o >> 5) * l + at(pb, h * kJb + (o & 31))] = y;
      T[(o >> 5) * (kJb + 1) + (o & 31)] = y;
    }
    if (a != b) {
      __syncthreads();
      for (int o = tid; o < kJp * kJb; o += kJacobiThreads)
        Mn[(size_t)at(pb, h * kJb + (o >> 6)) * l + at(pa, o & 63)] = T[(o & 63) * (kJb + 1) + (o >> 6)];
    }
  };

  int cur = 0, qb = 0;
  bool alive = grid_barrier(sy, arrived, &ok_s);
  int sweeps_done = 0;
  for (int sweep = 0; alive && sweep < kJacobiSweeps; ++sweep) {
    // ---- off-diagonal weight of M, as it is and with every entry beside its diagonal: per-CTA partial sums, then every CTA
    // adds them up in the same order
    {
      const float* M = cur ? M1 : M0;
      float* const inv = js;                                 // 1 / sqrt of the diagonal, floored
      float mx = 0.0f;
      for (int i = tid; i < l; i += kJacobiThreads) { inv[i] = __ldcg(M + (size_t)i * l + i); mx = fmaxf(mx, inv[i]); }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
      if (lane == 0) red_s[warp].x = mx;
      __syncthreads();
      mx = red_s[lane].x;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
      const float least = fmaxf(kJacobiFloor * mx, 1e-30f);
      for (int i = tid; i < l; i += kJacobiThreads) inv[i] = rsqrtf(fmaxf(inv[i], least));
      __syncthreads();
      float off = 0.0f, all = 0.0f, scaled = 0.0f;
      for (long long e = gtid; e < (long long)l * l; e += gstride) {
        const float v = __ldcg(M + e);
        const int i = (int)(e / l), j = (int)(e % l);
        all += v * v;
        if (i != j) {
          const float u = v * inv[i] * inv[j];
          off += v * v;
          scaled += u * u;
        }
      }
      auto total = [&]() {                                   // of the three over the CTA, in a fixed order; in thread 0
        auto fold = [&]() {
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) {
            off += __shfl_xor_sync(0xffffffffu, off, o);
            all += __shfl_xor_sync(0xffffffffu, all, o);
            scaled += __shfl_xor_sync(0xffffffffu, scaled, o);
          }
        };
        fold();
        if (lane == 0) red_s[warp] = make_float3(off, all, scaled);
        __syncthreads();
        if (warp == 0) {
          off = red_s[lane].x; all = red_s[lane].y; scaled = red_s[lane].z;
          fold();
        }
        __syncthreads();
      };
      total();
      if (tid == 0) partial[(sweep & 1) * nb + bid] = make_float4(off, all, scaled, 0.0f);
      alive = grid_barrier(sy, arrived, &ok_s);
      if (!alive) break;
      off = all = scaled = 0.0f;
      for (int b = tid; b < nb; b += kJacobiThreads) {
        const float4 v = __ldcg(partial + (sweep & 1) * nb + b);
        off += v.x; all += v.y; scaled += v.z;
      }
      total();
      if (tid == 0) done_s = (off <= kJacobiTol * all && scaled <= kJacobiScaledTol * kJacobiScaledTol * (float)l * (float)l) ? 1 : 0;
      __syncthreads();
      if (done_s) break;                                     // the same decision in every CTA
    }
    ++sweeps_done;
    const int items = npair * npair;                         // (pair, 64 columns of Pt)
    for (int t = 0; alive && t < nblk - 1; ++t) {
      const float* M = cur ? M1 : M0;
      float* Mn = cur ? M0 : M1;
      float* Q = Qg + (size_t)qb * npair * kJp * kJp;
      const float* Qprev = Qg + (size_t)(qb ^ 1) * npair * kJp * kJp;
      if (bid < npair) {
        for (int k = bid; k < npair; k += nb) solve_pair(M, tournament_pair(k, t, nblk), t == 0, Q + (size_t)k * kJp * kJp);
      } else if (t > 0) {
        for (int it = bid - npair; it < items; it += nb - npair)
          rotate_vectors(tournament_pair(it / npair, t - 1, nblk), (it % npair) * kJp, Qprev + (size_t)(it / npair) * kJp * kJp);
      }
      alive = grid_barrier(sy, arrived, &ok_s);
      if (!alive) break;
      for (int it = bid; it < npair * (npair + 1); it += nb) {   // pieces (a <= b, h)
        const int h = it & 1;
        int a = 0, rest = it >> 1;
        while (rest >= npair - a) { rest -= npair - a; ++a; }
        rotate_matrix(M, Mn, a, a + rest, h, t, Q);
      }
      alive = grid_barrier(sy, arrived, &ok_s);
      cur ^= 1;
      qb ^= 1;
    }
    if (!alive) break;
    for (int it = bid; it < items; it += nb)
      rotate_vectors(tournament_pair(it / npair, nblk - 2, nblk), (it % npair) * kJp,
                     Qg + ((size_t)(qb ^ 1) * npair + it / npair) * kJp * kJp);
  }
  if (bid == 0 && tid == 0) sy.abort[1] = (unsigned)sweeps_done;   // diagnostic: sweeps that ran
  if (alive && cur == 1) {                                   // the callers read buffer 0
    for (long long e = gtid; e < (long long)l * l; e += gstride) M0[e] = __ldcg(M1 + e);
  }
}

// The r largest eigenvalues (ties to the lower index) and their eigenvectors as the rows of Ps (r x l); sigma =
// sqrt(lambda).  One warp per eigenvalue.  Pb, if wanted: the rows again as bf16, what that rounding leaves out, and half of
// the first.
constexpr int kSelectWarps = 8;
__global__ void __launch_bounds__(kSelectWarps * 32)
eig_select_kernel(const float* __restrict__ M, const float* __restrict__ Pt, int l, int r, float* __restrict__ Ps,
                  __nv_bfloat16* __restrict__ Pb, float* __restrict__ sigma) {
  const int lane = threadIdx.x & 31, i = blockIdx.x * kSelectWarps + (threadIdx.x >> 5);
  if (i >= l) return;
  const float li = M[(size_t)i * l + i];
  int rk = 0;
  for (int j = lane; j < l; j += 32) {
    const float lj = M[(size_t)j * l + j];
    rk += (lj > li || (lj == li && j < i)) ? 1 : 0;
  }
  rk = __reduce_add_sync(0xffffffffu, rk);
  if (rk >= r) return;
  if (lane == 0 && sigma) sigma[rk] = sqrtf(fmaxf(li, 0.0f));
  for (int j = lane; j < l; j += 32) {
    const float v = Pt[(size_t)i * l + j];
    const size_t at = (size_t)rk * l + j;
    Ps[at] = v;
    if (Pb) {
      const __nv_bfloat16 hi = __float2bfloat16(v);
      Pb[at] = hi;
      Pb[(size_t)r * l + at] = __float2bfloat16(v - __bfloat162float(hi));
      Pb[(size_t)2 * r * l + at] = __float2bfloat16(0.5f * __bfloat162float(hi));
    }
  }
}

// V = Z Ps^T (N x r, fp32), rounded to bf16: row-major (if Vb is not null), and as the per-layer matrices B [G][r][d], B[g][m][j] = V[g d + j][m].
// 64 x 64 tiles, 256 threads, 4 x 4 outputs per thread, chunks of 32 k.
__global__ void __launch_bounds__(256)
ritz_vectors_kernel(const float* __restrict__ Z, const float* __restrict__ Ps, int l, int r, int d, __nv_bfloat16* __restrict__ Vb,
                    __nv_bfloat16* __restrict__ B) {
  __shared__ __align__(16) float As[32][68], Bs[32][68];
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int n0 = blockIdx.y * 64, m0 = blockIdx.x * 64;
  const int fr = tid >> 3, fc = (tid & 7) * 4;         // staged rows fr, fr + 32; 4 k
  float4 pa[2], pb[2];
  auto fetch = [&](int k0) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      pa[h] = *reinterpret_cast<const float4*>(Z + (size_t)(n0 + fr + 32 * h) * l + k0 + fc);
      const int m = m0 + fr + 32 * h;
      pb[h] = m < r ? *reinterpret_cast<const float4*>(Ps + (size_t)m * l + k0 + fc) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    }
  };
  float acc[4][4] = {};
  fetch(0);
  for (int k0 = 0; k0 < l; k0 += 32) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int row = fr + 32 * h;
      As[fc][row] = pa[h].x; As[fc + 1][row] = pa[h].y; As[fc + 2][row] = pa[h].z; As[fc + 3][row] = pa[h].w;
      Bs[fc][row] = pb[h].x; Bs[fc + 1][row] = pb[h].y; Bs[fc + 2][row] = pb[h].z; Bs[fc + 3][row] = pb[h].w;
    }
    __syncthreads();
    if (k0 + 32 < l) fetch(k0 + 32);
#pragma unroll
    for (int kk = 0; kk < 32; ++kk) {
      const float4 av = *reinterpret_cast<const float4*>(&As[kk][ty * 4]), bv = *reinterpret_cast<const float4*>(&Bs[kk][tx * 4]);
      const float a[4] = {av.x, av.y, av.z, av.w}, b[4] = {bv.x, bv.y, bv.z, bv.w};
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int n = n0 + ty * 4 + i, g = n / d, j = n - g * d;
#pragma unroll
    for (int x = 0; x < 4; ++x) {
      const int m = m0 + tx * 4 + x;
      if (m < r) {
        const __nv_bfloat16 v = __float2bfloat16(acc[i][x]);
        if (Vb) Vb[(size_t)n * r + m] = v;
        B[((size_t)g * r + m) * d + j] = v;
      }
    }
  }
}

}  // namespace

namespace {

// out = the sum of n_part arrays of n4 float4, in a fixed order.
__global__ void __launch_bounds__(256)
sum_parts_kernel(const float4* __restrict__ part, int n_part, long long n4, float4* __restrict__ out) {
  const long long i = (long long)blockIdx.x * 256 + threadIdx.x;
  if (i >= n4) return;
  float4 v = part[i];
  for (int z = 1; z < n_part; ++z) {
    const float4 u = part[(long long)z * n4 + i];
    v.x += u.x; v.y += u.y; v.z += u.z; v.w += u.w;
  }
  out[i] = v;
}

// M = (S + S^T) / 2 for the sum S of the partial products part [n_part][l][l], in a fixed order.
__global__ void symmetrize_kernel(const float* __restrict__ part, int n_part, float* __restrict__ M, int l) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= l * l) return;
  const int i = e / l, j = e % l;
  if (i > j) return;
  float a = 0.0f, b = 0.0f;
  for (int z = 0; z < n_part; ++z) { a += part[((size_t)z * l + i) * l + j]; b += part[((size_t)z * l + j) * l + i]; }
  const float v = 0.5f * (a + b);
  M[(size_t)i * l + j] = v;
  M[(size_t)j * l + i] = v;
}

// k of a product, all parts: whole blocks of 64 per part
int gemm_k(int K, int parts) { return parts == 1 ? K : parts * ((K + 63) & ~63); }
int gemm_splits(int M, int N, int K, int most);

struct ClfPlan {
  int T, Tp, N, r, l, q;
  int gram_split, gram_rows;                                 // row ranges of a Gram matrix and rows of each
  int u_split, ritz_split;                                   // K ranges of U = X^T Y and of the Ritz matrix
  size_t off_flags, off_zb, off_yt, off_yl, off_up, off_u, off_z, off_part, off_g, off_rt, off_w, off_iv, off_m, off_p, off_ps, off_vb, off_cs, off_m2,
      off_q, total;
};

size_t align_up(size_t x) { return (x + 255) & ~(size_t)255; }

bool make_plan(const xkv_clf_config* c, ClfPlan* p) {
  p->T = c->T; p->Tp = (c->T + 7) & ~7; p->N = c->G * c->d; p->r = c->r; p->q = c->power_iters;
  const int over = c->oversample > 0 ? c->oversample : 32;
  p->l = (c->r + over + 63) & ~63;
  if (p->l > p->N) p->l = p->N & ~63;
  if (p->l < c->r || p->l < 64 || p->l / 2 > kJacobiMaxPairs) return false;
  size_t o = 0;
  p->off_flags = o; o = align_up(o + 256);
  p->off_zb = o; o = align_up(o + (size_t)2 * p->N * p->l * 2);  // Z as two bf16 matrices, one below the other
  p->off_yt = o; o = align_up(o + (size_t)p->l * p->Tp * 2);
  p->off_yl = o; o = align_up(o + (size_t)p->l * p->Tp * 2);        // twice what the rounding of W leaves out
  p->u_split = gemm_splits(p->N, p->l, p->T, 8);
  p->off_up = o; if (p->u_split > 1) o = align_up(o + (size_t)p->u_split * p->N * p->l * 4);   // partial sums of U
  p->off_u = o; o = align_up(o + (size_t)p->N * p->l * 4);
  p->off_z = o; o = align_up(o + (size_t)p->N * p->l * 4);
  // row ranges so that the lower 64 x 64 tiles of the Gram matrix fill the SMs about twice
  const int tiles = (p->l / 64) * (p->l / 64 + 1) / 2;
  const int fill = 2 * kPlanSms / tiles;
  p->gram_split = fill < 1 ? 1 : fill > 8 ? 8 : fill;
  p->gram_rows = ((p->N + p->gram_split - 1) / p->gram_split + 31) & ~31;
  p->gram_split = (p->N + p->gram_rows - 1) / p->gram_rows;
  p->ritz_split = gemm_splits(p->l, p->l, gemm_k(p->T, 2), 16);
  const size_t part_words = p->gram_split * 2 > p->ritz_split ? p->gram_split * 2 : p->ritz_split;
  p->off_part = o; o = align_up(o + part_words * p->l * p->l * 4);   // partial Gram matrices (fp64) / Ritz matrices (fp32)
  p->off_g = o; o = align_up(o + (size_t)p->l * p->l * 8);      // the Gram matrix, factorised in place of its tiles, fp64
  p->off_rt = o; o = align_up(o + (size_t)p->l * p->l * 8);     // the identity under elimination, tiles transposed
  p->off_w = o; o = align_up(o + (size_t)p->l * p->l * 8);      // the factor's inverse
  p->off_iv = o; o = align_up(o + (size_t)p->l * kCholNb * 8);  // inverses of its diagonal blocks
  p->off_m = o; o = align_up(o + (size_t)p->l * p->l * 4);
  p->off_p = o; o = align_up(o + (size_t)p->l * p->l * 4);
  p->off_ps = o; o = align_up(o + (size_t)p->l * p->r * 4);
  p->off_vb = o; o = align_up(o + (size_t)p->N * p->r * 2);
  p->off_cs = o; o = align_up(o + (size_t)2 * 1024 * 16);           // per-CTA partial sums of the Jacobi convergence check
  p->off_m2 = o; o = align_up(o + (size_t)p->l * p->l * 4);      // second buffers of the one-kernel Jacobi sweeps
  p->off_q = o; o = align_up(o + (size_t)2 * p->l * kJp * 4);    // rotation products of the block pairs, two rounds
  p->total = o;
  return true;
}

int check_clf_config(const xkv_clf_config* c) {
  if (!c || c->struct_size != sizeof(xkv_clf_config)) return XKV_ERR_INVALID_ARG;
  if (c->T < 1 || c->T >= (1 << 24) || c->G < 1 || c->d < 8 || c->r < 8 || c->power_iters < 0 || c->power_iters > 8 ||
      c->oversample < 0)
    return XKV_ERR_INVALID_ARG;
  if (c->r % 8 || (c->G * (long long)c->d) % 64 || c->G * (long long)c->d > (1 << 20)) return XKV_ERR_INVALID_ARG;
  if (c->r > c->G * c->d) return XKV_ERR_INVALID_ARG;
  return XKV_OK;
}

// An operand of a product: a matrix [rows][cols] with a row pitch (elements); its columns are k if it is K-major, else its
// rows are.
struct GemmOperand {
  const void* p;
  int rows, cols, pitch;
};
struct GemmOut {
  float* f;                 // either may be null
  __nv_bfloat16* b;
  long long ld;
  __nv_bfloat16* lo = nullptr;   // transposed results only: twice what b's rounding leaves out
};

// Further parts of a product, laid out like the first: a (b + b2) + a3 b3.
struct GemmParts {
  const void *b2 = nullptr, *a3 = nullptr, *b3 = nullptr;
};

template <bool TRANS, bool AK, bool BK, bool LO, int MB, int BN>
cudaError_t launch_gemm_bn(GemmOperand a, GemmOperand b, const GemmParts& more, int splits, GemmOut c, unsigned int* flags, int device,
                           cudaStream_t s) {
  const int M = AK ? a.rows : a.cols, N = BK ? b.rows : b.cols, K = AK ? a.cols : a.rows;
  const int parts = more.a3 ? 3 : more.b2 ? 2 : 1, k_all = gemm_k(K, parts), k_part = k_all / parts;
  CUtensorMap ma, mb, mb2, ma3, mb3;
  if (!encode_bf16_map(&ma, a.p, (uint64_t)a.rows, (uint64_t)a.cols, (uint64_t)a.pitch, AK ? 128 * MB : 64) ||
      !encode_bf16_map(&mb, b.p, (uint64_t)b.rows, (uint64_t)b.cols, (uint64_t)b.pitch, BK ? BN : 64) ||
      !encode_bf16_map(&mb2, parts > 1 ? more.b2 : b.p, (uint64_t)b.rows, (uint64_t)b.cols, (uint64_t)b.pitch, BK ? BN : 64) ||
      !encode_bf16_map(&ma3, parts > 2 ? more.a3 : a.p, (uint64_t)a.rows, (uint64_t)a.cols, (uint64_t)a.pitch, AK ? 128 * MB : 64) ||
      !encode_bf16_map(&mb3, parts > 2 ? more.b3 : b.p, (uint64_t)b.rows, (uint64_t)b.cols, (uint64_t)b.pitch, BK ? BN : 64))
    return cudaErrorInvalidValue;
  const size_t smem = 1024 + (size_t)gemm_stages<MB, BN>() * gemm_stage_bytes<MB, BN>();
  cudaError_t e = ensure_dyn_smem<clf_gemm_kernel<TRANS, AK, BK, LO, MB, BN>>(smem, device);
  if (e != cudaSuccess) return e;
  const int k_per = ((k_all + splits - 1) / splits + 63) & ~63;
  const dim3 tiles((N + BN - 1) / BN, (M + 128 * MB - 1) / (128 * MB), splits);
  int sms = 0;
  if ((e = device_sms(device, &sms)) != cudaSuccess) return e;
  const long long n_tiles = (long long)tiles.x * tiles.y * tiles.z;
  const unsigned grid = (unsigned)(n_tiles < sms ? n_tiles : sms);        // one CTA per SM (shared and tensor memory)
  clf_gemm_kernel<TRANS, AK, BK, LO, MB, BN><<<grid, gemm_threads<MB>(), smem, s>>>(ma, mb, mb2, ma3, mb3, M, N, k_part, k_all, k_per, c.f, c.b, c.lo, c.ld, tiles,
                                                                               flags);
  count_launch(kFamClf);
  return cudaGetLastError();
}

// Tile width: the one that pads N least (the widest on a tie): 576 columns are three tiles of 192, 512 are two of 256.
int gemm_bn(int N) {
  auto padded = [&](int bn) { return (long long)((N + bn - 1) / bn) * bn; };
  int bn = 256;
  if (padded(192) < padded(bn)) bn = 192;
  if (padded(128) < padded(bn)) bn = 128;
  return bn;
}
// Two accumulators unless that pads M by more than an eighth.
int gemm_mb(int M) { return ((M + 255) & ~255) * 8LL <= ((M + 127) & ~127) * 9LL ? 2 : 1; }

template <bool TRANS, bool AK, bool BK, bool LO = false>
cudaError_t launch_gemm(GemmOperand a, GemmOperand b, int splits, GemmOut c, unsigned int* flags, int device, cudaStream_t s,
                        GemmParts more = {}) {
  const int bn = gemm_bn(BK ? b.rows : b.cols);
  if (gemm_mb(AK ? a.rows : a.cols) == 2) {
    if (bn == 256) return launch_gemm_bn<TRANS, AK, BK, LO, 2, 256>(a, b, more, splits, c, flags, device, s);
    if (bn == 192) return launch_gemm_bn<TRANS, AK, BK, LO, 2, 192>(a, b, more, splits, c, flags, device, s);
    return launch_gemm_bn<TRANS, AK, BK, LO, 2, 128>(a, b, more, splits, c, flags, device, s);
  }
  if (bn == 256) return launch_gemm_bn<TRANS, AK, BK, LO, 1, 256>(a, b, more, splits, c, flags, device, s);
  if (bn == 192) return launch_gemm_bn<TRANS, AK, BK, LO, 1, 192>(a, b, more, splits, c, flags, device, s);
  return launch_gemm_bn<TRANS, AK, BK, LO, 1, 128>(a, b, more, splits, c, flags, device, s);
}

// K ranges that bring a product's tiles to about one per SM, none of them empty or shorter than 1024.
int gemm_splits(int M, int N, int K, int most) {
  const int mb = gemm_mb(M) * 128, bn = gemm_bn(N);
  const long long tiles = (long long)((M + mb - 1) / mb) * ((N + bn - 1) / bn);
  long long sp = kPlanSms / tiles;
  if (sp > most) sp = most;
  if (sp > K / 1024) sp = K / 1024;
  if (sp < 1) sp = 1;
  const int k_per = (int)(((K + sp - 1) / sp + 63) & ~63);
  return (K + k_per - 1) / k_per;
}

template <auto Kernel>
cudaError_t launch_cooperative(int grid, int threads, size_t smem, void** args, int device, cudaStream_t s) {
  cudaError_t e = ensure_dyn_smem<Kernel>(smem, device);
  if (e != cudaSuccess) return e;
  count_launch(kFamClf);
  return cudaLaunchCooperativeKernel((const void*)Kernel, dim3(grid), dim3(threads), args, smem, s);
}

}  // namespace

int clf_rank_l(const xkv_clf_config* c, int* l) {
  int st = check_clf_config(c);
  if (st != XKV_OK) return st;
  ClfPlan p;
  if (!make_plan(c, &p)) return XKV_ERR_UNSUPPORTED;
  *l = p.l;
  return XKV_OK;
}

int clf_workspace_bytes(const xkv_clf_config* c, uint64_t* bytes) {
  int st = check_clf_config(c);
  if (st != XKV_OK) return st;
  ClfPlan p;
  if (!make_plan(c, &p)) return XKV_ERR_UNSUPPORTED;
  *bytes = p.total;
  return XKV_OK;
}

// Debug/test entry of the tensor-core product alone: C (M x N, fp32) = A B^T, A bf16 [K][M], B bf16 [N][K].
cudaError_t clf_gemm(const void* a, const void* b, int M, int N, int K, float* C, unsigned int* flags, int device, cudaStream_t s) {
  return launch_gemm<false, false, true>({a, K, M, M}, {b, N, K, K}, 1, {C, nullptr, N}, flags, device, s);
}

static std::atomic<unsigned> g_clf_inject{0};
void clf_set_fault_injection(unsigned mask) { g_clf_inject.store(mask, std::memory_order_relaxed); }

int clf_factorize(const xkv_clf_config* c, const void* X, const void* omega, void* workspace, uint64_t workspace_bytes,
                  void* A_out, void* B_out, float* sigma, int device, cudaStream_t s) {
  int st = check_clf_config(c);
  if (st != XKV_OK) return st;
  ClfPlan p;
  if (!make_plan(c, &p)) return XKV_ERR_UNSUPPORTED;
  if (workspace_bytes < p.total) return XKV_ERR_INVALID_ARG;
  uint8_t* w = (uint8_t*)workspace;
  unsigned int* flags = (unsigned int*)(w + p.off_flags);
  __nv_bfloat16* Zb = (__nv_bfloat16*)(w + p.off_zb);
  __nv_bfloat16* Yt = (__nv_bfloat16*)(w + p.off_yt);
  float* U = (float*)(w + p.off_u);
  float* Z = (float*)(w + p.off_z);
  double* part = (double*)(w + p.off_part);
  double* Gm = (double*)(w + p.off_g);
  double* Rt = (double*)(w + p.off_rt);
  double* W = (double*)(w + p.off_w);
  double* Iv = (double*)(w + p.off_iv);
  float* Mm = (float*)(w + p.off_m);
  float* Pm = (float*)(w + p.off_p);
  float* Ps = (float*)(w + p.off_ps);
  __nv_bfloat16* Vb = (__nv_bfloat16*)(w + p.off_vb);
  const int N = p.N, r = p.r, T = p.T;
  int l = p.l, sms = 0;
  cudaError_t e = device_sms(device, &sms);
  if (e == cudaSuccess) e = cudaMemsetAsync(flags, 0, 256, s);
  if (e == cudaSuccess) e = cudaMemcpyAsync(Zb, omega, (size_t)N * l * 2, cudaMemcpyDeviceToDevice, s);
  // Y = X Z (stored as Y^T)  and  U = X^T Y
  auto product_y = [&]() { return launch_gemm<true, true, false>({X, T, N, N}, {Zb, N, l, l}, 1, {nullptr, Yt, p.Tp}, flags, device, s); };
  auto product_u = [&]() -> cudaError_t {
    float* out = p.u_split > 1 ? (float*)(w + p.off_up) : U;
    cudaError_t e2 = launch_gemm<false, false, true>({X, T, N, N}, {Yt, l, T, p.Tp}, p.u_split, {out, nullptr, l}, flags, device, s);
    if (e2 != cudaSuccess || p.u_split == 1) return e2;
    const long long n4 = (long long)N * l / 4;
    sum_parts_kernel<<<(unsigned)((n4 + 255) / 256), 256, 0, s>>>((const float4*)out, p.u_split, n4, (float4*)U);
    count_launch(kFamClf);
    return cudaGetLastError();
  };
  // Z = orth(U) by shifted Cholesky QR, the Gram matrix accumulated, factorised and inverted in fp64: its condition
  // number is the square of the iterate's, which after a multiplication by X^T X spans the whole range between the
  // largest singular value and the noise floor.  A pass divides the condition number by up to shift^-1/2; U is stored
  // in fp32, so its own is below 1e9 and the fp64 Gram matrix carries a shift of 1e-11 safely (its rounding errors are
  // below 1e-13).  One pass leaves an iterate well conditioned, which is all that the next multiplication needs; the last
  // iterate takes three and is orthonormal to fp32 rounding.  (Shifts that start at 1e-4 need two and five passes for a
  // worse subspace: residual 1.088 instead of 1.081 of the optimum.)
  constexpr double kShift = 1e-11;
  const int nbk = l / kCholNb, n_tiles = nbk * (nbk + 1) / 2;
  const int chol_grid = sms < (n_tiles > 32 ? n_tiles : 32) ? sms : (n_tiles > 32 ? n_tiles : 32);
  unsigned chol_arrived = 0;
  const unsigned injected = g_clf_inject.load(std::memory_order_relaxed);
  auto grid_sync = [&](int count, unsigned mask) {                     // the words were zeroed with the flag block above
    const bool inject = (injected & mask) != 0u;
    return GridSync{flags, flags + count, flags + 10, inject ? 1024u : kGridSpinLimit, inject ? 1u : 0u};
  };
  auto cholqr = [&](int passes) -> cudaError_t {                       // an odd number of passes ends in Z
    float* in = U;
    float* out = Z;
    for (int pass = 0; pass < passes; ++pass) {
      gram_kernel<<<dim3((l / 64) * (l / 64 + 1) / 2, p.gram_split), 256, 0, s>>>(in, part, N, l, p.gram_rows);
      double shift = kShift;
      int n_part = p.gram_split;
      GridSync sy = grid_sync(12, XKV_INJECT_CLF_CHOLESKY);
      void* args[] = {&part, &n_part, &Gm, &Rt, &Iv, &W, &l, &shift, &chol_arrived, &sy};
      cudaError_t e2 = launch_cooperative<chol_inverse_kernel>(chol_grid, kCholThreads, 0, args, device, s);
      if (e2 != cudaSuccess) return e2;
      chol_arrived += (unsigned)chol_grid * (unsigned)(nbk + 1);       // barriers of one factorisation
      tri_product_kernel<<<dim3((N + 63) / 64, l / 64), 256, 0, s>>>(in, W, out, Zb, N, l);
      count_launch(kFamClf, 2);
      float* t = in; in = out; out = t;
    }
    return cudaGetLastError();
  };
  for (int it = 0; it <= p.q && e == cudaSuccess; ++it) {
    e = product_y();
    if (e == cudaSuccess) e = product_u();
    if (e == cudaSuccess) e = cholqr(it == p.q ? 3 : 1);
  }
  // Rayleigh-Ritz: W = X Z, M = W^T W (= Z^T X^T X Z), its eigenvectors by Jacobi.  M is that of the fp32 Z whose
  // combinations become V, so neither Z nor W may enter rounded to bf16.  A column of Z in the noise floor, rounded, holds
  // 2^-9 of the largest singular values: error of M_ij relative to sqrt(M_ii M_jj), rms, 1e-2 with the rounded Z on both
  // sides, 3e-3 as Z^T X^T (X Z_bf16), 1e-5 this way.  The rounding of W averages out over the rows, unless a few of them
  // hold most of the weight (sigma_1 of a cache with one row a thousand times the others: off by 3.7e-4 with W rounded on
  // both sides, 1.5e-4 on one).  With W = H + L the symmetric part of H^T (H + 2 L) is M up to L^T L.
  __nv_bfloat16* Yl = (__nv_bfloat16*)(w + p.off_yl);
  // A = X V = W P from the W that is there already, H (P1 + P2) + (2 L) (P1 / 2) with P = P1 + P2 in bf16 too (they take the
  // place of V_bf16 in the workspace): 3 l instead of N terms a sum, and without the rounding of V in them (what P1 + P2
  // leaves out is 2^-17).  131072 x 4096, r = 512, the call and the reconstruction behind it 7554 -> 7338 us.  Residual over
  // the optimum of that rank, 2048 to 20000 rows, five shapes: 1.0299-1.0456 -> 1.0293-1.0432; with an outlier row or column
  // 1.17-7.7 -> 1.16-7.1.  Where 3 l is not less than N the product with V_bf16 is the shorter one.
  const bool from_w = 3 * l < N;
  if (e == cudaSuccess) e = launch_gemm<true, true, false, true>({X, T, N, N}, {Zb, N, l, l}, 1, {nullptr, Yt, p.Tp, Yl}, flags, device, s, {Zb + (size_t)N * l});
  if (e == cudaSuccess) e = launch_gemm<false, true, true>({Yt, l, T, p.Tp}, {Yt, l, T, p.Tp}, p.ritz_split, {(float*)part, nullptr, l}, flags, device, s, {Yl});
  if (e == cudaSuccess) {
    symmetrize_kernel<<<(l * l + 255) / 256, 256, 0, s>>>((const float*)part, p.ritz_split, Mm, l);
    float* M2 = (float*)(w + p.off_m2);
    float* Qm = (float*)(w + p.off_q);
    float4* partial = (float4*)(w + p.off_cs);
    GridSync sy = grid_sync(8, XKV_INJECT_CLF_BARRIER);
    unsigned arrived = 0;
    void* args[] = {&Mm, &M2, &Pm, &Qm, &l, &partial, &arrived, &sy};
    e = launch_cooperative<jacobi_block_kernel>(sms, kJacobiThreads, kJacobiSmem, args, device, s);
  }
  if (e == cudaSuccess) {
    eig_select_kernel<<<(l + kSelectWarps - 1) / kSelectWarps, kSelectWarps * 32, 0, s>>>(Mm, Pm, l, r, Ps, from_w ? Vb : nullptr, sigma);
    ritz_vectors_kernel<<<dim3((r + 63) / 64, N / 64), 256, 0, s>>>(Z, Ps, l, r, c->d, from_w ? nullptr : Vb, (__nv_bfloat16*)B_out);
    count_launch(kFamClf, 3);
    e = cudaGetLastError();
  }
  // A = X V, stored [T][r]
  if (e == cudaSuccess && from_w)
    e = launch_gemm<false, false, true>({Yt, l, T, p.Tp}, {Vb, r, l, l}, 1, {nullptr, (__nv_bfloat16*)A_out, r}, flags, device, s,
                                        {Vb + (size_t)r * l, Yl, Vb + (size_t)2 * r * l});
  else if (e == cudaSuccess)
    e = launch_gemm<false, true, false>({X, T, N, N}, {Vb, N, r, r}, 1, {nullptr, (__nv_bfloat16*)A_out, r}, flags, device, s);
  if (e != cudaSuccess) { set_cuda_error(e); (void)cudaGetLastError(); return XKV_ERR_CUDA; }
  return XKV_OK;
}

}  // namespace xkv
