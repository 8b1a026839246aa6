// Landmark-guided top-k chunk selection (App. B.1, Algorithm 2) in two kernels, a scan and a top-k:
//   score_pool_kernel   lines 2-3: streams every landmark once (HBM bound), fp32 scores in the canonical order, max-pool over the
//                       query heads of each KV head;
//   score_bound_kernel  the same with scores by mma.sync and a bound on their error, for more than four heads per KV head and calls
//                       of some size (launch_select_dev has the line);
//   topk_pivot_kernel   lines 1, 4, 5: the k_ch largest pooled scores of up to 32768 chunks by a filtered list (ties to the lowest
//                       chunk index), united with the outlier chunks, ascending, expanded to token rows; of scores with a bound
//                       those around the cut are worked out again in the canonical order;
//   topk_kernel         the same for longer contexts, by radix select over all keys.
#include <cuda.h>
#include <math.h>

#include <mutex>

#include "xkv_internal.cuh"
#include "xkv_ptx.cuh"

namespace xkv {

namespace {

constexpr int kScoreRows = kLandmarkBoxRows;   // landmark rows (chunks) per CTA
constexpr int kScoreThreads = 32;    // two rows per thread
constexpr uint32_t kWaitLimit = 1u << 22;

using namespace ptx;

// Bounded wait: returns false if the phase did not complete within `limit` polls.
__device__ __forceinline__ bool mbar_wait_bounded(uint32_t bar, uint32_t parity, uint32_t limit = kWaitLimit) {
  for (uint32_t i = 0; i < limit; ++i) {
    if (mbar_try_wait(bar, parity)) return true;
  }
  return false;
}
__device__ __forceinline__ uint4 lds128(uint32_t addr) {
  uint4 v;
  asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr));
  return v;
}

// Order-preserving map float -> uint32 (larger float = larger key), with -0 folded onto +0.
__device__ __forceinline__ uint32_t score_key(float f) {
  uint32_t u = __float_as_uint(f);
  if (u == 0x80000000u) u = 0u;
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

// One pass over the staged tile for HB query heads; returns per-row max of the scaled scores.
template <int DH, int HB>
__device__ __forceinline__ void score_pass(uint32_t tile, const float* __restrict__ qs, int row0, float s,
                                           float& best0, float& best1) {
  float acc0[HB], acc1[HB];
#pragma unroll
  for (int h = 0; h < HB; ++h) { acc0[h] = 0.0f; acc1[h] = 0.0f; }
  const uint32_t sw = (uint32_t)(row0 & 7);
  const uint32_t a0 = tile + (uint32_t)row0 * 128u;
  const uint32_t a1 = a0 + (uint32_t)kScoreThreads * 128u;
#pragma unroll 4
  for (int cc = 0; cc < DH / 8; ++cc) {
    const uint32_t off = (uint32_t)(cc >> 3) * (kScoreRows * 128u) + ((((uint32_t)cc & 7u) ^ sw) << 4);
    const uint4 va = lds128(a0 + off);
    const uint4 vb = lds128(a1 + off);
    const uint32_t wa[4] = {va.x, va.y, va.z, va.w};
    const uint32_t wb[4] = {vb.x, vb.y, vb.z, vb.w};
    float qv[HB][8];
#pragma unroll
    for (int h = 0; h < HB; ++h) {
      const float4 q0 = *reinterpret_cast<const float4*>(qs + h * DH + cc * 8);
      const float4 q1 = *reinterpret_cast<const float4*>(qs + h * DH + cc * 8 + 4);
      qv[h][0] = q0.x; qv[h][1] = q0.y; qv[h][2] = q0.z; qv[h][3] = q0.w;
      qv[h][4] = q1.x; qv[h][5] = q1.y; qv[h][6] = q1.z; qv[h][7] = q1.w;
    }
    // element by element (ascending i, the canonical order of every sum), all heads and both rows per element: the
    // 2 * HB multiply-adds of an element are independent of one another
#pragma unroll
    for (int w = 0; w < 4; ++w) {
      const float xa0 = __uint_as_float(wa[w] << 16), xb0 = __uint_as_float(wb[w] << 16);
      const float xa1 = __uint_as_float(wa[w] & 0xffff0000u), xb1 = __uint_as_float(wb[w] & 0xffff0000u);
#pragma unroll
      for (int h = 0; h < HB; ++h) {
        acc0[h] = fmaf(qv[h][2 * w], xa0, acc0[h]);
        acc1[h] = fmaf(qv[h][2 * w], xb0, acc1[h]);
      }
#pragma unroll
      for (int h = 0; h < HB; ++h) {
        acc0[h] = fmaf(qv[h][2 * w + 1], xa1, acc0[h]);
        acc1[h] = fmaf(qv[h][2 * w + 1], xb1, acc1[h]);
      }
    }
  }
#pragma unroll
  for (int h = 0; h < HB; ++h) {
    best0 = fmaxf(best0, acc0[h] * s);
    best1 = fmaxf(best1, acc1[h] * s);
  }
}

// grid.x = ceil(n_c / kScoreRows) tiles, grid.y = (layers in call) * batch * H_kv problems.
template <int DH, int HMAX>
__global__ void __launch_bounds__(kScoreThreads)
score_pool_kernel(const __grid_constant__ CUtensorMap tmap, GroupDev dev, const __nv_bfloat16* __restrict__ q,
                  int l0) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t bar_storage;
  const uint32_t tile = (smem_u32(smem_raw) + 1023u) & ~1023u;
  float* qs = reinterpret_cast<float*>(smem_raw + (tile - smem_u32(smem_raw)) + (DH / 64) * kScoreRows * 128);
  const uint32_t bar = smem_u32(&bar_storage);

  const int g = blockIdx.y % dev.H_kv;
  const int b = (blockIdx.y / dev.H_kv) % dev.batch;
  const int l = l0 + blockIdx.y / (dev.H_kv * dev.batch);
  const int j0 = blockIdx.x * kScoreRows;
  const long long prob_lm = ((long long)b * dev.G + l) * dev.H_kv + g;       // landmark order
  const long long prob_out = ((long long)l * dev.batch + b) * dev.H_kv + g;  // [G][batch][H_kv] order

  // fault injection (tests of the give-up path): no load is issued, so the wait below must run into its limit
  const bool no_load = (dev.inject & XKV_INJECT_SCAN_NO_LOAD) != 0u;
  // A handle's landmarks are constant while the handle is used (the caller's contract), so their loads may start
  // before the kernel launched before this one has finished; the queries may come from that kernel and are
  // read after the dependency wait.  Without a handle (the allocation-free entry point) nothing is known about
  // the landmarks, and the loads wait too.
  const bool early = dev.lm_const != 0;
  if (!early) grid_dependency_wait();
  if (threadIdx.x == 0) {          // the thread that initialises the barrier also issues the loads: nothing to wait for
    mbar_init(bar, 1);
    fence_mbar_init();
    if (!no_load) {
      mbar_expect_tx(bar, (uint32_t)((DH / 64) * kScoreRows * 128));
      const int y = (int)(prob_lm * dev.n_c + j0);
      // every landmark is read once per call: first in line for eviction, so that the stream does not push the
      // pooled scores (written below, read by the top-k) and the gathered basis rows out of L2
      const uint64_t pol = l2_policy_evict_first();
#pragma unroll
      for (int bx = 0; bx < DH / 64; ++bx) tma_load_2d_hint(tile + bx * kScoreRows * 128, &tmap, bx * 64, y, bar, pol);
    }
  }
  if (early) grid_dependency_wait();
  grid_dependency_launch();
  // queries of this KV head, widened to fp32 while the landmarks are in flight
  const __nv_bfloat16* qg = q + (((long long)l * dev.batch + b) * dev.H_q + (long long)g * dev.n_rep) * DH;
  // (all the 16-byte loads of a lane are issued before the first is used: one trip to L2, not one per element)
  {
    const uint4* qv = reinterpret_cast<const uint4*>(qg);
    const int n_pieces = dev.n_rep * (DH / 8);
    constexpr int kMaxPieces = kMaxRep * (DH / 8) / kScoreThreads;   // at most kMaxRep query heads per KV head
    uint4 u[kMaxPieces];
#pragma unroll
    for (int i = 0; i < kMaxPieces; ++i) {
      const int pc = threadIdx.x + i * kScoreThreads;
      u[i] = pc < n_pieces ? qv[pc] : make_uint4(0u, 0u, 0u, 0u);
    }
#pragma unroll
    for (int i = 0; i < kMaxPieces; ++i) {
      const int pc = threadIdx.x + i * kScoreThreads;
      if (pc < n_pieces) {
        float4 a, b;
        a.x = __uint_as_float(u[i].x << 16); a.y = __uint_as_float(u[i].x & 0xffff0000u);
        a.z = __uint_as_float(u[i].y << 16); a.w = __uint_as_float(u[i].y & 0xffff0000u);
        b.x = __uint_as_float(u[i].z << 16); b.y = __uint_as_float(u[i].z & 0xffff0000u);
        b.z = __uint_as_float(u[i].w << 16); b.w = __uint_as_float(u[i].w & 0xffff0000u);
        *reinterpret_cast<float4*>(qs + pc * 8) = a;
        *reinterpret_cast<float4*>(qs + pc * 8 + 4) = b;
      }
    }
  }
  __syncthreads();

  if (!mbar_wait_bounded(bar, 0, no_load ? 1024u : kWaitLimit)) {
    if (threadIdx.x == 0) atomicOr(dev.flags, XKV_FLAG_TIMEOUT);
    // The boxes may still be on their way into this CTA's shared memory, which the next CTA on the SM would
    // inherit: stay for a second (again bounded) wait before giving the memory up.
    if (!no_load) (void)mbar_wait_bounded(bar, 0);
    return;
  }
  float best0 = -INFINITY, best1 = -INFINITY;
  const int row0 = threadIdx.x;
  // heads in passes of HMAX: a pass reads the tile once for all its heads.  The kernel for up to four heads per
  // KV head is kept apart from the wider one: its code is smaller, and the scan is sensitive to that.
  for (int h0 = 0; h0 < dev.n_rep; h0 += HMAX) {
    const int hb = min(HMAX, dev.n_rep - h0);
    const float* qh = qs + h0 * DH;
    if constexpr (HMAX == 8) {
      if (hb == 8) { score_pass<DH, 8>(tile, qh, row0, dev.sel_scale, best0, best1); continue; }
      if (hb == 7) { score_pass<DH, 7>(tile, qh, row0, dev.sel_scale, best0, best1); continue; }
      if (hb == 6) { score_pass<DH, 6>(tile, qh, row0, dev.sel_scale, best0, best1); continue; }
      if (hb == 5) { score_pass<DH, 5>(tile, qh, row0, dev.sel_scale, best0, best1); continue; }
    }
    if (hb == 4) score_pass<DH, 4>(tile, qh, row0, dev.sel_scale, best0, best1);
    else if (hb == 3) score_pass<DH, 3>(tile, qh, row0, dev.sel_scale, best0, best1);
    else if (hb == 2) score_pass<DH, 2>(tile, qh, row0, dev.sel_scale, best0, best1);
    else score_pass<DH, 1>(tile, qh, row0, dev.sel_scale, best0, best1);
  }
  // the pooled scores are handed on as order-preserving integer keys (what the top-k compares)
  uint32_t* dst = reinterpret_cast<uint32_t*>(dev.pooled) + prob_out * dev.n_c;
  if (j0 + row0 < dev.n_c) dst[j0 + row0] = score_key(best0);
  if (j0 + row0 + kScoreThreads < dev.n_c) dst[j0 + row0 + kScoreThreads] = score_key(best1);
}

// ---- The scan with more than four query heads per KV head: tensor-core scores and their error bound.
// Only the index sets leave the selection, so a score has to be the canonical one only where it decides something: the
// scores here carry an error of at most E, and topk_pivot_kernel scores the few chunks within 2 E of the cut again in the
// canonical order.  score_pool_kernel is bound by the shared-memory pipe with that many heads (14 query loads of four cycles
// for 112 multiply-adds per 8 dimensions at seven); here a landmark leaves shared memory once, as the fragments of
// mma.sync.m16n8k16, whose eight columns are the heads, and the queries stay in registers.  What bounds it is the landmarks.
// mma.sync and not tcgen05: 0.1 TFLOP in all, and a warp keeps its own tile without tensor memory or a second barrier.
//
// The bound.  The products are exact in fp32.  With S = sum_i |q_i l_i| of a row and a head the canonical chain of d_h <= 128
// multiply-adds is off by at most 128 2^-24 S, d_h / 16 steps of 17 terms and a sum, each cut off below 2^-23 of the largest
// at worst, by at most 144 2^-23 S, and scaling adds one rounding to either: less than 0.82 2^-15 S together (S itself, from
// the tensor core too, is short by less than 2^-15 of it).  S comes from the same fragments without their signs, its largest
// value in a tile is written beside the scores, and E is that of the largest of the problem.  (|q|_1 max |l| in its place needs no
// further products, but is a hundred times larger where one channel or row stands out, and the band with it.  Selections of
// 65536 rows, seven heads, 128 problems, with that -> with S: Gaussian landmarks 47.0 -> 46.5 us, a channel of 300 72 -> 49, one
// row in a hundred a hundred times as long 75 -> 52, one element of 1000 144 -> 48, of 3000 575 -> 53; canonical scan 68.)
constexpr float kScoreBound = 1.0f / 32768.0f;

__device__ __forceinline__ void ldmatrix_x4(uint32_t (&r)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void mma_16816(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// grid as above.  NT: groups of eight heads.  tile_sum [problem][tile]: bits of the tile's largest S (a NaN above everything;
// 0: all its rows or all the queries are zero, and so is every score).
template <int DH, int NT>
__global__ void __launch_bounds__(kScoreThreads)
score_bound_kernel(const __grid_constant__ CUtensorMap tmap, GroupDev dev, const __nv_bfloat16* __restrict__ q, int l0) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t bar_storage;
  constexpr int KS = DH / 16;
  const uint32_t tile = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const uint32_t bar = smem_u32(&bar_storage);
  const int lane = threadIdx.x, g8 = lane >> 2, t = lane & 3;

  const int g = blockIdx.y % dev.H_kv;
  const int b = (blockIdx.y / dev.H_kv) % dev.batch;
  const int l = l0 + blockIdx.y / (dev.H_kv * dev.batch);
  const int j0 = blockIdx.x * kScoreRows;
  const long long prob_lm = ((long long)b * dev.G + l) * dev.H_kv + g;       // landmark order
  const long long prob_out = ((long long)l * dev.batch + b) * dev.H_kv + g;  // [G][batch][H_kv] order

  // loads ahead of the dependency wait, fault injection, limits: as in score_pool_kernel
  const bool no_load = (dev.inject & XKV_INJECT_SCAN_NO_LOAD) != 0u;
  const bool early = dev.lm_const != 0;
  if (!early) grid_dependency_wait();
  if (lane == 0) {
    mbar_init(bar, 1);
    fence_mbar_init();
    if (!no_load) {
      mbar_expect_tx(bar, (uint32_t)((DH / 64) * kScoreRows * 128));
      const int y = (int)(prob_lm * dev.n_c + j0);
      const uint64_t pol = l2_policy_evict_first();
#pragma unroll
      for (int bx = 0; bx < DH / 64; ++bx) tma_load_2d_hint(tile + bx * kScoreRows * 128, &tmap, bx * 64, y, bar, pol);
    }
  }
  if (early) grid_dependency_wait();
  grid_dependency_launch();
  // this lane's fragments of the queries: head 8 n + g8, dimensions 16 ks + 2 t, + 1 and those 8 on (heads beyond n_rep: zero)
  const __nv_bfloat16* qg = q + (((long long)l * dev.batch + b) * dev.H_q + (long long)g * dev.n_rep) * DH;
  uint32_t qf[NT][KS][2];
#pragma unroll
  for (int n = 0; n < NT; ++n) {
    const int h = 8 * n + g8;
    const uint32_t* qh = reinterpret_cast<const uint32_t*>(qg + (size_t)h * DH) + t;
#pragma unroll
    for (int ks = 0; ks < KS; ++ks)
#pragma unroll
      for (int x = 0; x < 2; ++x) qf[n][ks][x] = h < dev.n_rep ? qh[ks * 8 + x * 4] : 0u;
  }
  __syncwarp();

  if (!mbar_wait_bounded(bar, 0, no_load ? 1024u : kWaitLimit)) {
    if (lane == 0) atomicOr(dev.flags, XKV_FLAG_TIMEOUT);
    if (!no_load) (void)mbar_wait_bounded(bar, 0);
    return;
  }
  // lane i hands ldmatrix the address of row i % 16, dimensions 8 (i / 16) of a 16 x 16 piece
  const uint32_t arow = (uint32_t)(lane & 15), ahalf = (uint32_t)(lane >> 4);
  float keep[2] = {0.0f, 0.0f};                            // rows 16 t + g8 and 16 t + 8 + g8
  uint32_t big = 0u;                                       // largest S
#pragma unroll
  for (int m = 0; m < kScoreRows / 16; ++m) {
    const uint32_t row = (uint32_t)(16 * m) + arow, sw = row & 7u;
    float acc[NT][4], sum[NT][4];
#pragma unroll
    for (int n = 0; n < NT; ++n)
#pragma unroll
      for (int i = 0; i < 4; ++i) acc[n][i] = sum[n][i] = 0.0f;
#pragma unroll
    for (int ks = 0; ks < KS; ++ks) {
      uint32_t a[4], mag[4];
      ldmatrix_x4(a, tile + (uint32_t)(ks >> 2) * (kScoreRows * 128u) + row * 128u + ((((uint32_t)(ks & 3) * 2u + ahalf) ^ sw) << 4));
#pragma unroll
      for (int i = 0; i < 4; ++i) mag[i] = a[i] & 0x7fff7fffu;
#pragma unroll
      for (int n = 0; n < NT; ++n) {
        mma_16816(acc[n], a, qf[n][ks][0], qf[n][ks][1]);
        mma_16816(sum[n], mag, qf[n][ks][0] & 0x7fff7fffu, qf[n][ks][1] & 0x7fff7fffu);
      }
    }
    // (the box runs on beyond the last chunk, into the next problem's rows: they do not count)
#pragma unroll
    for (int n = 0; n < NT; ++n)
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (j0 + 16 * m + 8 * (i >> 1) + g8 < dev.n_c) big = max(big, __float_as_uint(sum[n][i]) & 0x7fffffffu);
    // columns 2 t, 2 t + 1 of rows g8 (acc 0, 1) and g8 + 8 (acc 2, 3): maximum over the heads that exist
    float best[2] = {-INFINITY, -INFINITY};
#pragma unroll
    for (int n = 0; n < NT; ++n)
#pragma unroll
      for (int x = 0; x < 2; ++x)
        if (8 * n + 2 * t + x < dev.n_rep) {
          best[0] = fmaxf(best[0], acc[n][x] * dev.sel_scale);
          best[1] = fmaxf(best[1], acc[n][2 + x] * dev.sel_scale);
        }
#pragma unroll
    for (int o = 1; o < 4; o <<= 1) {
      best[0] = fmaxf(best[0], __shfl_xor_sync(0xffffffffu, best[0], o));
      best[1] = fmaxf(best[1], __shfl_xor_sync(0xffffffffu, best[1], o));
    }
    if (t == m) { keep[0] = best[0]; keep[1] = best[1]; }
  }
  static_assert(kScoreRows == 64, "four lanes of a row, four pieces of 16 rows");
  uint32_t* dst = reinterpret_cast<uint32_t*>(dev.pooled) + prob_out * dev.n_c;
#pragma unroll
  for (int x = 0; x < 2; ++x) {
    const int j = j0 + 16 * t + 8 * x + g8;
    if (j < dev.n_c) dst[j] = score_key(keep[x]);
  }
  big = __reduce_max_sync(0xffffffffu, big);
  if (big == 0u) {
    // zero, or so small that the products are lost: only the first is exact (all rows of the box are looked at)
    uint32_t any_l = 0u, any_q = 0u;
    for (uint32_t off = (uint32_t)lane * 16u; off < (uint32_t)((DH / 64) * kScoreRows * 128); off += 512u) {
      const uint4 v = lds128(tile + off);
      any_l |= v.x | v.y | v.z | v.w;
    }
    any_l &= 0x7fff7fffu;
#pragma unroll
    for (int n = 0; n < NT; ++n)
#pragma unroll
      for (int ks = 0; ks < KS; ++ks) any_q |= (qf[n][ks][0] | qf[n][ks][1]) & 0x7fff7fffu;
    if (__any_sync(0xffffffffu, any_l != 0u) && __any_sync(0xffffffffu, any_q != 0u)) big = 1u;
  }
  if (lane == 0) dev.tile_sum[prob_out * gridDim.x + blockIdx.x] = big;
}

// ---------------------------------------------------------------------------------------------

constexpr int kTopkThreads = 1024;
constexpr int kTopkItems = 16;    // consecutive chunks per thread and super-block
constexpr int kTopkBins = 2048;   // histogram bins per radix pass
constexpr int kTopkCand = 256;    // at most this many keys are ranked against one another directly

// Keys of this thread's 16 consecutive chunks of one super-block (0 beyond n_c; callers mask by index).
// sign == 0: the array already holds keys (the landmark scan writes them); else it holds floats and the key is
// that of sign * value.
template <int ITEMS>
__device__ __forceinline__ void load_keys(const float* __restrict__ S, int j0, int n_c, float sign, uint32_t (&key)[ITEMS]) {
  const bool keyed = sign == 0.0f;
  if (j0 + ITEMS <= n_c && ((n_c & 3) == 0)) {
    const float4* p = reinterpret_cast<const float4*>(S + j0);
#pragma unroll
    for (int i = 0; i < ITEMS / 4; ++i) {
      const float4 v = p[i];
      const float f[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int e = 0; e < 4; ++e) key[4 * i + e] = keyed ? __float_as_uint(f[e]) : score_key(f[e] * sign);
    }
  } else {
#pragma unroll
    for (int i = 0; i < ITEMS; ++i) {
      const float f = (j0 + i < n_c) ? S[j0 + i] : 0.0f;
      key[i] = (j0 + i < n_c) ? (keyed ? __float_as_uint(f) : score_key(f * sign)) : 0u;
    }
  }
}

// One CTA per (layer, sequence, KV head).  grid.x = problems of the call.
// Exact k_ch-th largest key by a radix select whose bins subdivide the range that still contains it
// (first the [min, max] range of all keys, then the chosen bin, ...: at most three 11-bit passes), followed
// by an ordered compaction.  The keys are read again in every pass (they come from L2).
__global__ void __launch_bounds__(kTopkThreads)
topk_kernel(GroupDev dev, int l0, int k_ch, int k_cap, const int32_t* __restrict__ outliers, int n_out, float sign,
            int32_t* __restrict__ sel_idx, int32_t* __restrict__ sel_cnt) {
  __shared__ __align__(16) uint32_t hist[kTopkBins];
  __shared__ uint32_t warp_tot[kTopkThreads / 32];
  __shared__ uint32_t warp_min[kTopkThreads / 32], warp_max[kTopkThreads / 32];
  __shared__ uint32_t sh_a, sh_b, sh_c;

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int per_layer = dev.batch * dev.H_kv;
  const long long prob = (long long)l0 * per_layer + blockIdx.x;     // [G][batch][H_kv] order
  const float* __restrict__ S = dev.pooled + prob * dev.n_c;
  int32_t* __restrict__ out = sel_idx + prob * k_cap;
  const int n_c = dev.n_c, c = dev.c, T = dev.T;
  const int super = kTopkThreads * kTopkItems;
  const bool out_vec = (reinterpret_cast<uintptr_t>(out) & 15u) == 0;   // 16-byte stores of the row ids

  grid_dependency_wait();                      // the pooled scores come from the kernel launched before
  grid_dependency_launch();

  uint32_t thr = 0, need_eq = 0;
  const bool all = (k_ch >= n_c);
  if (!all) {
    // ---- range of the keys
    uint32_t kmin = 0xffffffffu, kmax = 0u;
    for (int base = 0; base < n_c; base += super) {
      uint32_t key[kTopkItems];
      const int j0 = base + tid * kTopkItems;
      load_keys(S, j0, n_c, sign, key);
#pragma unroll
      for (int i = 0; i < kTopkItems; ++i) {
        if (j0 + i < n_c) { kmin = min(kmin, key[i]); kmax = max(kmax, key[i]); }
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      kmin = min(kmin, __shfl_xor_sync(0xffffffffu, kmin, o));
      kmax = max(kmax, __shfl_xor_sync(0xffffffffu, kmax, o));
    }
    if (lane == 0) { warp_min[warp] = kmin; warp_max[warp] = kmax; }
    __syncthreads();
    kmin = warp_min[lane]; kmax = warp_max[lane];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      kmin = min(kmin, __shfl_xor_sync(0xffffffffu, kmin, o));
      kmax = max(kmax, __shfl_xor_sync(0xffffffffu, kmax, o));
    }
    // ---- radix passes over the window [lo, lo + span]
    uint32_t lo = kmin, span = kmax - kmin, need = (uint32_t)k_ch;
    for (;;) {
      const int bits = 32 - __clz(span);                      // span < 2^bits
      const int sh = bits > 11 ? bits - 11 : 0;
      for (int i = tid; i < kTopkBins; i += kTopkThreads) hist[i] = 0;
      __syncthreads();
      for (int base = 0; base < n_c; base += super) {
        uint32_t key[kTopkItems];
        const int j0 = base + tid * kTopkItems;
        load_keys(S, j0, n_c, sign, key);
#pragma unroll
        for (int i = 0; i < kTopkItems; ++i) {
          const uint32_t rel = key[i] - lo;
          if (j0 + i < n_c && key[i] >= lo && rel <= span) atomicAdd(&hist[rel >> sh], 1u);
        }
      }
      __syncthreads();
      // suffix counts from the top bin down: thread t owns bins 2t, 2t+1
      const uint32_t h0 = hist[2 * tid], h1 = hist[2 * tid + 1];
      const uint32_t mine = h0 + h1;
      uint32_t suf = mine;                                     // inclusive over higher lanes of the warp
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t v = __shfl_down_sync(0xffffffffu, suf, o);
        if (lane + o < 32) suf += v;
      }
      if (lane == 0) warp_tot[warp] = suf;
      __syncthreads();
      if (warp == 0) {
        const uint32_t t = warp_tot[lane];
        uint32_t ws = t;                                       // inclusive over higher warps
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const uint32_t v = __shfl_down_sync(0xffffffffu, ws, o);
          if (lane + o < 32) ws += v;
        }
        warp_tot[lane] = ws - t;                               // keys in bins of higher warps
      }
      __syncthreads();
      const uint32_t above = warp_tot[warp] + (suf - mine);    // keys in bins above 2t+1
      if (above < need && above + mine >= need) {              // exactly one thread
        if (above + h1 >= need) { sh_a = 2 * tid + 1; sh_b = need - above; sh_c = h1; }
        else { sh_a = 2 * tid; sh_b = need - above - h1; sh_c = h0; }
      }
      __syncthreads();
      const uint32_t bsel = sh_a, in_bin = sh_c;
      need = sh_b;
      lo += bsel << sh;
      span = min(span - (bsel << sh), (sh ? (1u << sh) : 1u) - 1u);
      __syncthreads();
      if (sh == 0) { thr = lo; need_eq = need; break; }
      if (in_bin <= (uint32_t)kTopkCand) {
        // Few keys are left in the window: collect them (in any order) and rank them against one another.
        // The `need`-th largest of them is the threshold; need_eq = how many keys equal to it are still wanted.
        uint32_t* cand = hist;
        if (tid == 0) sh_a = 0;
        __syncthreads();
        for (int base = 0; base < n_c; base += super) {
          uint32_t key[kTopkItems];
          const int j0 = base + tid * kTopkItems;
          load_keys(S, j0, n_c, sign, key);
          // this thread's candidates as a bit mask; the warp reserves room for all of its candidates with one atomic
          uint32_t cm = 0;
#pragma unroll
          for (int i = 0; i < kTopkItems; ++i) {
            if (j0 + i < n_c && key[i] >= lo && key[i] - lo <= span) cm |= 1u << i;
          }
          const uint32_t mine_c = (uint32_t)__popc(cm);
          if (__any_sync(0xffffffffu, cm != 0u)) {
            uint32_t inc = mine_c;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
              const uint32_t v = __shfl_up_sync(0xffffffffu, inc, o);
              if (lane >= o) inc += v;
            }
            uint32_t wbase = 0;
            if (lane == 31) wbase = atomicAdd(&sh_a, inc);
            wbase = __shfl_sync(0xffffffffu, wbase, 31);
            uint32_t at = wbase + inc - mine_c;
#pragma unroll
            for (int i = 0; i < kTopkItems; ++i) {
              if ((cm >> i) & 1u) cand[at++] = key[i];
            }
          }
        }
        __syncthreads();
        const uint32_t n_cand = sh_a;                          // == in_bin
        __syncthreads();
        if ((uint32_t)tid < n_cand) {
          const uint32_t mykey = cand[tid];
          uint32_t gt = 0, eq = 0;
          const uint32_t n4 = n_cand & ~3u;
          const uint4* c4 = reinterpret_cast<const uint4*>(cand);
#pragma unroll 4
          for (uint32_t i = 0; i < n4; i += 4) {
            const uint4 v = c4[i >> 2];
            gt += (v.x > mykey ? 1u : 0u) + (v.y > mykey ? 1u : 0u) + (v.z > mykey ? 1u : 0u) + (v.w > mykey ? 1u : 0u);
            eq += (v.x == mykey ? 1u : 0u) + (v.y == mykey ? 1u : 0u) + (v.z == mykey ? 1u : 0u) + (v.w == mykey ? 1u : 0u);
          }
          for (uint32_t i = n4; i < n_cand; ++i) {
            const uint32_t c2 = cand[i];
            gt += c2 > mykey ? 1u : 0u;
            eq += c2 == mykey ? 1u : 0u;
          }
          if (gt < need && need <= gt + eq) { sh_a = mykey; sh_b = need - gt; }   // equal keys write the same pair
        }
        __syncthreads();
        thr = sh_a;
        need_eq = sh_b;
        __syncthreads();
        break;
      }
    }
  }

  // Ordered compaction: chunk j is taken if key > thr, or key == thr and fewer than need_eq equal
  // keys precede it, or (Algorithm 2 line 5) it is one of the head's static outlier chunks.  Positions follow
  // ascending j.
  __shared__ uint32_t obits[kTopkThreads * kTopkItems / 32];   // outlier chunks of the current super-block
  __shared__ uint32_t sh_last_taken;
  // packed (low 16 bits, high 16 bits) exclusive prefix over the CTA in thread order; the total goes to sh_a
  auto block_scan = [&](uint32_t mine) -> uint32_t {
    uint32_t inc = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t v = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += v;
    }
    if (lane == 31) warp_tot[warp] = inc;
    __syncthreads();
    if (warp == 0) {
      const uint32_t t = warp_tot[lane];
      uint32_t ti = t;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t v = __shfl_up_sync(0xffffffffu, ti, o);
        if (lane >= o) ti += v;
      }
      warp_tot[lane] = ti - t;                      // exclusive prefix of warp totals
      if (lane == 31) sh_a = ti;                    // super-block total
    }
    __syncthreads();
    return inc - mine + warp_tot[warp];
  };
  auto write_chunk = [&](uint32_t pos, int j) {
    const int rows = min(c, T - j * c);
    if (c == 8 && rows == 8 && out_vec) {
      int4* o4 = reinterpret_cast<int4*>(out + (size_t)pos * 8);
      o4[0] = make_int4(j * 8, j * 8 + 1, j * 8 + 2, j * 8 + 3);
      o4[1] = make_int4(j * 8 + 4, j * 8 + 5, j * 8 + 6, j * 8 + 7);
    } else {
      for (int t = 0; t < rows; ++t) out[(size_t)pos * c + t] = j * c + t;
    }
  };
  const int32_t* outl = nullptr;                    // this problem's outlier chunk ids
  if (n_out > 0) {
    outl = outliers + (size_t)prob * (size_t)n_out;          // [G][batch][H_kv][n_out], like sel_idx
    if (tid == 0) sh_last_taken = 0;
  }
  uint32_t run_gt = 0, run_eq = 0;                  // totals of the super-blocks already done
  uint32_t run_taken = 0;                           // chunks written so far (outlier path)
  uint32_t last_key = 0;
  for (int base = 0; base < n_c; base += super) {
    const int j0 = base + tid * kTopkItems;
    uint32_t gtm = 0, eqm = 0;                      // bit i set: item i is > / == thr
    if (all) {
#pragma unroll
      for (int i = 0; i < kTopkItems; ++i) if (j0 + i < n_c) gtm |= 1u << i;
    } else {
      uint32_t key[kTopkItems];
      load_keys(S, j0, n_c, sign, key);
#pragma unroll
      for (int i = 0; i < kTopkItems; ++i) {
        if (j0 + i < n_c) {
          gtm |= (key[i] > thr ? 1u : 0u) << i;
          eqm |= (key[i] == thr ? 1u : 0u) << i;
          if (j0 + i == n_c - 1) last_key = key[i];
        }
      }
    }
    const uint32_t mine = (uint32_t)__popc(gtm) | ((uint32_t)__popc(eqm) << 16);
    const uint32_t excl = block_scan(mine);
    const uint32_t tot1 = sh_a;
    uint32_t gt_before = run_gt + (excl & 0xffffu);
    uint32_t eq_before = run_eq + (excl >> 16);
    if (n_out == 0) {
      // Only a few percent of the chunks are taken.  Output position of a taken chunk = taken chunks before it.
      // If the super-block's taken chunks fit the list (the histogram's memory, free by now), their ids go there
      // first and the whole CTA then writes the rows, consecutive threads to consecutive words; else every thread
      // writes the rows of its own chunks.
      const uint32_t blk_gt = tot1 & 0xffffu, blk_eq = tot1 >> 16;
      const uint32_t eq_room = need_eq > run_eq ? need_eq - run_eq : 0u;        // equal keys this super-block may still take
      const uint32_t blk_taken = blk_gt + min(blk_eq, eq_room);
      const uint32_t pos0 = run_gt + min(run_eq, need_eq);                       // chunks written by earlier super-blocks
      const bool listed = blk_taken <= (uint32_t)kTopkBins;
      uint32_t m = gtm | eqm;
      while (m) {
        const int i = __ffs(m) - 1;
        m &= m - 1;
        const uint32_t below = (1u << i) - 1u;
        const uint32_t g_b = gt_before + (uint32_t)__popc(gtm & below), e_b = eq_before + (uint32_t)__popc(eqm & below);
        const bool is_gt = (gtm >> i) & 1u;
        if (is_gt || e_b < need_eq) {
          const uint32_t pos = g_b + min(e_b, need_eq);
          if (listed) hist[pos - pos0] = (uint32_t)(j0 + i); else write_chunk(pos, j0 + i);
        }
      }
      if (listed) {
        __syncthreads();
        if (c == 8) {
          for (uint32_t w = (uint32_t)tid; w < blk_taken * 8u; w += kTopkThreads) {
            const int row = (int)hist[w >> 3] * 8 + (int)(w & 7u);
            if (row < T) out[(size_t)pos0 * 8 + w] = row;
          }
        } else {
          for (uint32_t w = (uint32_t)tid; w < blk_taken * (uint32_t)c; w += kTopkThreads) {
            const uint32_t e = w / (uint32_t)c, t = w - e * (uint32_t)c;
            const int row = (int)hist[e] * c + (int)t;
            if (row < T) out[(size_t)pos0 * c + w] = row;
          }
        }
      }
    } else {
      // membership in the top-k first, then the union with the outlier chunks, then positions over the union
      uint32_t takem = 0;
#pragma unroll
      for (int i = 0; i < kTopkItems; ++i) {
        const bool is_gt = (gtm >> i) & 1u, is_eq = (eqm >> i) & 1u;
        if (is_gt || (is_eq && eq_before < need_eq)) takem |= 1u << i;
        gt_before += is_gt ? 1u : 0u;
        eq_before += is_eq ? 1u : 0u;
      }
      for (int w = tid; w < super / 32; w += kTopkThreads) obits[w] = 0u;
      __syncthreads();                                // also: everybody has read sh_a and warp_tot of the first scan
      const int hi = min(base + super, n_c);
      for (int o = tid; o < n_out; o += kTopkThreads) {
        const int jo = outl[o];
        if (jo >= base && jo < hi) atomicOr(&obits[(jo - base) >> 5], 1u << ((jo - base) & 31));
      }
      __syncthreads();
      static_assert(kTopkItems == 16, "two threads share one word of the outlier bitmap");
      takem |= (obits[tid >> 1] >> ((tid & 1) * 16)) & 0xffffu;
      const uint32_t excl2 = block_scan((uint32_t)__popc(takem));
      uint32_t pos = run_taken + excl2;
#pragma unroll
      for (int i = 0; i < kTopkItems; ++i) {
        if ((takem >> i) & 1u) {
          write_chunk(pos++, j0 + i);
          if (j0 + i == n_c - 1) sh_last_taken = 1u;
        }
      }
      run_taken += sh_a;
    }
    run_gt += tot1 & 0xffffu;
    run_eq += tot1 >> 16;
    __syncthreads();
  }
  // Row count: whole chunks unless the ragged last chunk was taken (it is then the last one).
  // Without outliers: k_ch chunks; the last chunk has the highest index, so it wins a tie only if every equal key fits.
  __shared__ uint32_t sh_last;                    // key of chunk n_c-1, published by the thread that owns it
  {
    const int owner = ((n_c - 1) % super) / kTopkItems;
    if (tid == owner) sh_last = last_key;
    __syncthreads();
  }
  int cnt;
  if (n_out == 0) {
    cnt = (all ? n_c : k_ch) * c;
    bool last_in = all;
    if (!all) last_in = sh_last > thr || (sh_last == thr && run_eq <= need_eq);
    if (last_in) cnt -= (n_c * c - T);
  } else {
    cnt = (int)run_taken * c;
    if (sh_last_taken) cnt -= (n_c * c - T);
  }
  for (int i = cnt + tid; i < k_cap; i += kTopkThreads) out[i] = -1;
  if (tid == 0 && sel_cnt) sel_cnt[prob] = cnt;
}


// ---------------------------------------------------------------------------------------------
// The same selection for n_c <= 32768 chunks, organised so that almost all of the work is done on a short list instead
// of on every key.  Latency bound: one CTA per problem on an otherwise idle chip, a chain of barriers; what counts is
// their number (eleven) and what lies between them.
//   1  every thread's keys (16-byte loads side by side), the maximum of each of its GPT groups
//   2  the k_ch-th largest group maximum, by one histogram, is a lower bound P of the k_ch-th largest key (at least k_ch
//      keys -- those maxima -- are >= it), and with k_ch a few percent of n_c only a few percent of the keys pass it
//   3  the keys >= P go to a list in shared memory (key, chunk index)
//   4  a histogram over the list finds the bin of the k_ch-th largest key; keys of higher bins are taken
//   5  the few keys of that bin are ranked against one another by (key, chunk index), which also settles ties: a warp
//      per candidate, its lanes holding the candidates in registers
//   6  membership is a bitmap over the chunks (united with the head's outlier chunks); its prefix popcounts give the
//      ascending output positions
// Bins of more than kTopkCand keys are subdivided; if all their keys are equal, the lowest chunk indices are taken from a
// second bitmap.  GPT = 0 disables the filter (P = the smallest key): chosen by the host when there are fewer groups than
// k_ch.  ITEMS = 16 keys per thread serve n_c <= 16384 chunks, ITEMS = 32 (keys read twice instead of held in registers)
// n_c <= 32768.  The result is identical to topk_kernel's for every input.
//
// BOUND: the keys are those of score_bound_kernel, off by at most E (see there).  The k_ch-th largest canonical score then
// lies within E of the k_ch-th largest key, so chunks more than 2 E above the bin of step 4 are taken and those more than 2 E
// below it are not; the band between is scored again in the canonical order and its keys take the place of the bin's.  Step 3
// lists down to P - 2 E.  With E = 0 (nothing but zeros) the keys are the canonical ones.  A band of more than kTopkCand chunks
// (that many scores equal to 2^-14 of S, or a score that is not finite somewhere, where E is infinite and the band everything)
// goes through the bins again, a chunk per thread on the problem's one SM (8192 chunks of one and the same score, 128 problems of
// seven heads: 201 us, a warp per chunk 663, the canonical scan with its top-k 75; 64 problems of sixteen heads and 16384 chunks
// 635, 1270 and 154).  Tiles of zeros are left out of that: the unused end of a context, 98 % zeros: 72 us, canonical 79.
// (With consecutive keys per thread, extrema by shuffles, a thread per candidate and separate scans for ties and
// positions, about 25 barriers: 32768 rows decoded layer by layer 129.4 us, 122.4 us with this form; 121873 rows 212.6 ->
// 193.6; 2048 rows 19.3 -> 17.6.)

// Bin (counted from the top) that holds the `need`-th largest of the keys counted in hist[0..kTopkBins), by a suffix sum
// over the bins; thread t of the TH owns the kTopkBins / TH bins from t * (kTopkBins / TH).  Results in sh[0] = bin,
// sh[1] = rank wanted inside the bin, sh[2] = keys in the bin.  Contains barriers: call it from all threads.
template <int TH>
__device__ __forceinline__ void find_bin(const uint32_t* hist, uint32_t need, uint32_t* warp_tot, uint32_t* sh, int tid) {
  constexpr int BPT = kTopkBins / TH, NWARP = TH / 32;
  static_assert(BPT >= 1 && BPT * TH == kTopkBins, "bins per thread");
  const int lane = tid & 31, warp = tid >> 5;
  uint32_t h[BPT];
  uint32_t mine = 0;
#pragma unroll
  for (int i = 0; i < BPT; ++i) { h[i] = hist[BPT * tid + i]; mine += h[i]; }
  const uint32_t wsum = __reduce_add_sync(0xffffffffu, mine);
  if (lane == 0) warp_tot[warp] = wsum;
  __syncthreads();
  // every warp works out which warp owns the bin; that warp goes on
  const uint32_t t = lane < NWARP ? warp_tot[lane] : 0u;
  const uint32_t higher = __reduce_add_sync(0xffffffffu, lane > warp ? t : 0u);     // keys in bins of higher warps
  if (higher < need && higher + wsum >= need) {
    uint32_t suf = mine;                                   // inclusive over higher lanes of the warp
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t v = __shfl_down_sync(0xffffffffu, suf, o);
      if (lane + o < 32) suf += v;
    }
    uint32_t acc = higher + suf - mine;                    // keys in bins above this thread's
    if (acc < need && acc + mine >= need) {                // exactly one thread
#pragma unroll
      for (int i = BPT - 1; i >= 0; --i) {
        if (acc < need && acc + h[i] >= need) { sh[0] = (uint32_t)(BPT * tid + i); sh[1] = need - acc; sh[2] = h[i]; }
        acc += h[i];
      }
    }
  }
  __syncthreads();
}

// float of a key (score_key's inverse but for -0)
__device__ __forceinline__ float key_score(uint32_t k) { return __uint_as_float((k & 0x80000000u) ? k ^ 0x80000000u : ~k); }

// The canonical pooled score of one landmark row, by a warp: lane h takes query head h.  q_s: bf16 queries in shared memory,
// 16-byte units, qu units to a head.
template <int DH>
__device__ __forceinline__ uint32_t canonical_key(const __nv_bfloat16* __restrict__ row, const uint4* __restrict__ q_s, int qu,
                                                  int n_rep, float scale, int lane) {
  const uint4* rv = reinterpret_cast<const uint4*>(row);
  uint4 v[DH / 8];
#pragma unroll
  for (int i = 0; i < DH / 8; ++i) v[i] = __ldg(rv + i);
  const uint4* qh = q_s + min(lane, n_rep - 1) * qu;
  float acc = 0.0f;
#pragma unroll
  for (int i = 0; i < DH / 8; ++i) {
    const uint4 qv = qh[i];
    const uint32_t lw[4] = {v[i].x, v[i].y, v[i].z, v[i].w}, qw[4] = {qv.x, qv.y, qv.z, qv.w};
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      acc = fmaf(__uint_as_float(qw[e] << 16), __uint_as_float(lw[e] << 16), acc);
      acc = fmaf(__uint_as_float(qw[e] & 0xffff0000u), __uint_as_float(lw[e] & 0xffff0000u), acc);
    }
  }
  // (the maximum of order-preserving keys is the key of the maximum; a NaN takes no part, as in fmaxf)
  return __reduce_max_sync(0xffffffffu, score_key(fmaxf(-INFINITY, acc * scale)));
}

// The same of one row by one thread: an element is loaded and widened once for eight heads.  q_f: fp32 queries in shared memory,
// dh to a head.
__device__ __forceinline__ uint32_t canonical_key_thread(const uint4* __restrict__ row, const float* __restrict__ q_f, int dh,
                                                      int n_rep, float scale) {
  float best = -INFINITY;
#pragma unroll 1
  for (int h0 = 0; h0 < n_rep; h0 += 8) {
    float acc[8];
#pragma unroll
    for (int h = 0; h < 8; ++h) acc[h] = 0.0f;
#pragma unroll 1
    for (int i = 0; i < dh / 8; i += 2) {
      const uint4 v0 = __ldg(row + i), v1 = __ldg(row + i + 1);
      const uint32_t lw[8] = {v0.x, v0.y, v0.z, v0.w, v1.x, v1.y, v1.z, v1.w};
      float x[16];
#pragma unroll
      for (int e = 0; e < 8; ++e) { x[2 * e] = __uint_as_float(lw[e] << 16); x[2 * e + 1] = __uint_as_float(lw[e] & 0xffff0000u); }
#pragma unroll
      for (int h = 0; h < 8; ++h) {
        if (h0 + h < n_rep) {
          const float4* qh = reinterpret_cast<const float4*>(q_f + (h0 + h) * dh + i * 8);
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const float4 qv = qh[e];
            acc[h] = fmaf(qv.w, x[4 * e + 3], fmaf(qv.z, x[4 * e + 2], fmaf(qv.y, x[4 * e + 1], fmaf(qv.x, x[4 * e], acc[h]))));
          }
        }
      }
    }
#pragma unroll
    for (int h = 0; h < 8; ++h) if (h0 + h < n_rep) best = fmaxf(best, acc[h] * scale);
  }
  return score_key(best);
}

// The listed chunks of a wide band (those with an entry other than 0) scored again, a thread per chunk, out of line: it is
// seldom taken.  q_s as above; q_f: room for them in fp32.  Chunks of a tile of zeros, the unused end of a context, have their
// key already.
__device__ __noinline__ void rescore_wide(uint32_t* __restrict__ list_key, const uint16_t* __restrict__ list_idx, int n_list,
                                          const __nv_bfloat16* __restrict__ rows, const uint32_t* __restrict__ tile_sum,
                                          const uint4* __restrict__ q_s, float* __restrict__ q_f, int n_rep, int dh, float scale) {
  const int pieces = dh / 8;
  if ((int)threadIdx.x < n_rep * pieces) {
    const uint4 v = q_s[threadIdx.x / pieces * (pieces + 1) + threadIdx.x % pieces];
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
    float* to = q_f + threadIdx.x * 8;
#pragma unroll
    for (int e = 0; e < 4; ++e) { to[2 * e] = __uint_as_float(w[e] << 16); to[2 * e + 1] = __uint_as_float(w[e] & 0xffff0000u); }
  }
  __syncthreads();
  for (int e = threadIdx.x; e < n_list; e += blockDim.x)
    if (list_key[e] != 0u && __ldcg(tile_sum + list_idx[e] / kScoreRows) != 0u)
      list_key[e] = canonical_key_thread(reinterpret_cast<const uint4*>(rows + (size_t)list_idx[e] * dh), q_f, dh, n_rep, scale);
}

template <int GPT, int ITEMS, int TH, bool BOUND>
__global__ void __launch_bounds__(TH, 1)
topk_pivot_kernel(GroupDev dev, int l0, int k_ch, int k_cap, const int32_t* __restrict__ outliers, int n_out, float sign,
                  const __nv_bfloat16* __restrict__ q, int32_t* __restrict__ sel_idx, int32_t* __restrict__ sel_cnt) {
  extern __shared__ __align__(16) uint8_t pivot_smem[];
  constexpr int kPivotListMax = TH * ITEMS;                              // every key may pass (all keys equal)
  constexpr int NW = kPivotListMax / 32;                                 // words of a bitmap
  static_assert(kPivotListMax <= 65536 && NW <= TH, "16-bit chunk index, one bitmap word per thread");
  uint32_t* list_key = reinterpret_cast<uint32_t*>(pivot_smem);                    // [kPivotListMax]; later the chunk list
  uint16_t* list_idx = reinterpret_cast<uint16_t*>(list_key + kPivotListMax);      // [kPivotListMax]
  __shared__ __align__(16) uint32_t hist0[kTopkBins], hist1[kTopkBins];
  __shared__ uint32_t take_w[NW], eq_w[NW];                                        // bitmaps over the chunks
  __shared__ uint32_t warp_tot[TH / 32], warp_eq[TH / 32];
  __shared__ uint32_t warp_min[TH / 32], warp_max[TH / 32];
  __shared__ unsigned long long cand_s[kTopkCand];                                 // (key, ~chunk index): larger = earlier
  __shared__ uint32_t sh[3];
  __shared__ uint32_t sh_n, sh_cand;
  __shared__ uint32_t warp_s[TH / 32];                                             // BOUND: largest S
  __shared__ uint32_t sh_sure;                                                     // BOUND: chunks taken without their canonical score

  constexpr int NWARP = TH / 32;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int per_layer = dev.batch * dev.H_kv;
  const long long prob = (long long)l0 * per_layer + blockIdx.x;     // [G][batch][H_kv] order
  const float* __restrict__ S = dev.pooled + prob * dev.n_c;
  int32_t* __restrict__ out = sel_idx + prob * k_cap;
  const int n_c = dev.n_c, c = dev.c, T = dev.T;
  constexpr int NG = GPT == 0 ? 1 : GPT;                               // group maxima kept per thread
  const bool all = (k_ch >= n_c);
  // chunk of this thread's key i: runs of four side by side where a row of scores starts on 16 bytes, else single ones
  const bool vec = (n_c & 3) == 0;
  auto chunk_of = [&](int i) { return vec ? (i >> 2) * (TH * 4) + tid * 4 + (i & 3) : i * TH + tid; };

  for (int i = tid; i < kTopkBins; i += TH) { hist0[i] = 0; hist1[i] = 0; }
  for (int w = tid; w < NW; w += TH) {
    const int first = w * 32;
    take_w[w] = !all ? 0u : first + 32 <= n_c ? 0xffffffffu : (first < n_c ? ((1u << (n_c - first)) - 1u) : 0u);
    eq_w[w] = 0u;
  }
  if (tid == 0) { sh_n = 0; sh_cand = 0; sh[0] = sh[1] = sh[2] = 0; sh_sure = 0; }
  grid_dependency_wait();                      // the pooled scores come from the kernel launched before
  grid_dependency_launch();
  const int pieces = dev.d_h / 8;              // 16-byte pieces of a query
  const long long head0 = (prob / dev.H_kv) * dev.H_q + (prob % dev.H_kv) * dev.n_rep;    // of this problem's queries
  uint4 q_piece = make_uint4(0u, 0u, 0u, 0u);
  if constexpr (BOUND) {
    static_assert(TH >= kMaxRep * 16, "a thread per piece of the queries");
    if (tid < dev.n_rep * pieces) q_piece = __ldg(reinterpret_cast<const uint4*>(q + head0 * dev.d_h) + tid);
  }
  bool ties = false;                           // the bin of the k_ch-th largest key holds equal keys only, and many of them
  uint32_t need = (uint32_t)k_ch;
  if (!all) {
    uint32_t key[ITEMS];
    // sign == 0: the array already holds keys (the landmark scan writes them); else the key is that of sign * value
    auto load = [&]() {
      if (vec) {
#pragma unroll
        for (int u = 0; u < ITEMS / 4; ++u) {
          const int j = u * (TH * 4) + tid * 4;
          const uint4 v = j < n_c ? __ldcg(reinterpret_cast<const uint4*>(S + j)) : make_uint4(0u, 0u, 0u, 0u);
          key[4 * u] = v.x; key[4 * u + 1] = v.y; key[4 * u + 2] = v.z; key[4 * u + 3] = v.w;
        }
      } else {
#pragma unroll
        for (int i = 0; i < ITEMS; ++i) {
          const int j = i * TH + tid;
          key[i] = j < n_c ? __float_as_uint(__ldcg(S + j)) : 0u;
        }
      }
      if (sign != 0.0f) {
#pragma unroll
        for (int i = 0; i < ITEMS; ++i) key[i] = chunk_of(i) < n_c ? score_key(__uint_as_float(key[i]) * sign) : 0u;
      }
    };
    load();
    if constexpr (BOUND) {
      const int n_t = (n_c + kScoreRows - 1) / kScoreRows;
      uint32_t big = 0u;
      for (int i = tid; i < n_t; i += TH) big = max(big, __ldcg(dev.tile_sum + prob * n_t + i));
      big = __reduce_max_sync(0xffffffffu, big);
      if (lane == 0) warp_s[warp] = big;
    }
    // ---- 1: maxima of the groups that hold a chunk, and their range (keys beyond the last chunk are 0)
    uint32_t gmax[NG], kmin = 0xffffffffu, kmax = 0u;
#pragma unroll
    for (int g = 0; g < NG; ++g) {
      uint32_t m = 0u;
#pragma unroll
      for (int i = g * (ITEMS / NG); i < (g + 1) * (ITEMS / NG); ++i) m = max(m, key[i]);
      gmax[g] = m;
      kmax = max(kmax, m);
      if (GPT != 0 && chunk_of(g * (ITEMS / NG)) < n_c) kmin = min(kmin, m);
    }
    if (GPT == 0) {
#pragma unroll
      for (int i = 0; i < ITEMS; ++i) if (chunk_of(i) < n_c) kmin = min(kmin, key[i]);
    }
    kmin = __reduce_min_sync(0xffffffffu, kmin);
    kmax = __reduce_max_sync(0xffffffffu, kmax);
    if (lane == 0) { warp_min[warp] = kmin; warp_max[warp] = kmax; }
    __syncthreads();
    kmin = __reduce_min_sync(0xffffffffu, lane < NWARP ? warp_min[lane] : 0xffffffffu);
    kmax = __reduce_max_sync(0xffffffffu, lane < NWARP ? warp_max[lane] : 0u);
    float E2 = 0.0f;                                       // BOUND: 2 E
    if constexpr (BOUND) {
      const float S = __uint_as_float(__reduce_max_sync(0xffffffffu, lane < NWARP ? warp_s[lane] : 0u));
      E2 = S == 0.0f ? 0.0f : S < 1e36f ? fmaf(2.0f * kScoreBound * dev.sel_scale, S, 1e-37f) : INFINITY;    // (also where S is NaN)
    }
    // ---- 2: pivot: lower edge of the bin that holds the k_ch-th largest group maximum
    uint32_t P = kmin;
    if (GPT != 0) {
      const int bits1 = 32 - __clz(kmax - kmin);
      const int sh1 = bits1 > 11 ? bits1 - 11 : 0;
#pragma unroll
      for (int g = 0; g < NG; ++g) if (chunk_of(g * (ITEMS / NG)) < n_c) atomicAdd(&hist0[(gmax[g] - kmin) >> sh1], 1u);
      __syncthreads();
      find_bin<TH>(hist0, (uint32_t)k_ch, warp_tot, sh, tid);
      P = kmin + (sh[0] << sh1);
    }
    uint32_t Pl = P;                                       // what is listed
    if constexpr (BOUND) {
      Pl = E2 < INFINITY ? min(P, score_key(__fadd_rd(key_score(P), -E2))) : 0u;
      if (tid < dev.n_rep * pieces) {                      // the queries, into the first histogram, whose work is done
        const int h = tid / pieces, u = tid - h * pieces;
        reinterpret_cast<uint4*>(hist0)[h * (pieces + 1) + u] = q_piece;
      }
      static_assert(kMaxRep * (16 + 1) * 4 <= kTopkBins, "queries in a histogram");
    }
    // ---- 3: the keys >= P, with their chunk index, to the list (one shared-memory atomic per warp)
    {
      if (ITEMS > 16) load();                              // 32 keys are not held across the barriers above: read them again
      uint32_t cm = 0;
#pragma unroll
      for (int i = 0; i < ITEMS; ++i) if (key[i] >= Pl && chunk_of(i) < n_c) cm |= 1u << i;
      const uint32_t mine_c = (uint32_t)__popc(cm);
      uint32_t inc = mine_c;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t v = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += v;
      }
      uint32_t wbase = 0;
      if (lane == 31 && inc != 0u) wbase = atomicAdd(&sh_n, inc);
      uint32_t at = __shfl_sync(0xffffffffu, wbase, 31) + inc - mine_c;
      if (cm != 0u) {
#pragma unroll
        for (int i = 0; i < ITEMS; ++i) {
          if ((cm >> i) & 1u) { list_key[at] = key[i]; list_idx[at] = (uint16_t)chunk_of(i); ++at; }
        }
      }
    }
    __syncthreads();
    const int n_list = (int)sh_n;                                      // >= k_ch
    // ---- 4: bins subdivide the window [lo, lo + span] that holds the k_ch-th largest key
    uint32_t lo = P, span = kmax - P, in_bin;
    auto narrow = [&](uint32_t most, bool again) {         // down to `most` keys, or equal ones
      for (;; again = true) {
        const int bits = 32 - __clz(span);                             // span < 2^bits
        const int shb = bits > 11 ? bits - 11 : 0;
        if (again) {
          for (int i = tid; i < kTopkBins; i += TH) hist1[i] = 0;
          __syncthreads();
        }
        for (int e = tid; e < n_list; e += TH) {
          const uint32_t rel = list_key[e] - lo;                       // keys below lo wrap to huge values
          if (rel <= span) atomicAdd(&hist1[rel >> shb], 1u);
        }
        __syncthreads();
        find_bin<TH>(hist1, need, warp_tot, sh, tid);
        const uint32_t bsel = sh[0];
        need = sh[1];
        in_bin = sh[2];
        lo += bsel << shb;
        span = min(span - (bsel << shb), (shb ? (1u << shb) : 1u) - 1u);
        if (shb == 0 || in_bin <= most) break;
        __syncthreads();                                               // sh is read before the next pass writes it
      }
    };
    const bool exact = !BOUND || E2 == 0.0f;
    narrow(exact ? (uint32_t)kTopkCand : (uint32_t)NWARP, false);
    bool ranked = false;                                   // the candidates are in cand_s already
    if (BOUND && !exact) {
      // chunks above the band are taken; those in it keep their entry and are listed (the first kTopkCand of them)
      // (at least the bin is in the band, whatever the keys are: fewer than k_ch chunks are above it, k_ch at or above its foot)
      const uint32_t above = E2 < INFINITY ? max(lo + span, score_key(__fadd_ru(key_score(lo + span), E2))) : 0xffffffffu;
      const uint32_t below = E2 < INFINITY ? min(lo, score_key(__fadd_rd(key_score(lo), -E2))) : 0u;
      const __nv_bfloat16* rows = dev.landmarks + ((prob / dev.H_kv % dev.batch * dev.G + prob / per_layer) * dev.H_kv + prob % dev.H_kv) * n_c * dev.d_h;
      auto exact_key = [&](uint32_t j) {
        const __nv_bfloat16* row = rows + (size_t)j * dev.d_h;
        const uint4* q_s = reinterpret_cast<const uint4*>(hist0);
        return dev.d_h == 128 ? canonical_key<128>(row, q_s, pieces + 1, dev.n_rep, dev.sel_scale, lane)
                              : canonical_key<64>(row, q_s, pieces + 1, dev.n_rep, dev.sel_scale, lane);
      };
      for (int e = tid; e < n_list; e += TH) {
        const uint32_t kk = list_key[e], j = list_idx[e];
        const bool sure = kk > above, band = !sure && kk >= below;
        if (sure) { atomicOr(&take_w[j >> 5], 1u << (j & 31u)); atomicAdd(&sh_sure, 1u); }
        if (band) {
          const uint32_t at = atomicAdd(&sh_cand, 1u);
          if (at < (uint32_t)kTopkCand) cand_s[at] = j;
        }
        // out of the band: 0, in it: not 0, whatever the key (the key of a score never is 0, but a scan that gave up leaves
        // what was there before)
        list_key[e] = band ? max(kk, 1u) : 0u;
      }
      __syncthreads();
      in_bin = sh_cand;                                    // with the chunks taken, at least k_ch
      need = (uint32_t)k_ch - sh_sure;
      ranked = in_bin <= (uint32_t)kTopkCand;
      if (ranked) {
        for (uint32_t e = (uint32_t)warp; e < in_bin; e += NWARP) {
          const uint32_t j = (uint32_t)cand_s[e], kk = exact_key(j);
          if (lane == 0) cand_s[e] = ((unsigned long long)kk << 32) | (0xffffffffu - j);
        }
      } else {
        static_assert(kMaxRep * 128 <= kTopkBins, "fp32 queries in a histogram");
        rescore_wide(list_key, list_idx, n_list, rows, dev.tile_sum + prob * ((n_c + kScoreRows - 1) / kScoreRows),
                     reinterpret_cast<const uint4*>(hist0), reinterpret_cast<float*>(hist1), dev.n_rep, dev.d_h, dev.sel_scale);
        __syncthreads();
        if (tid == 0) sh_cand = 0;
        lo = 1u; span = 0xfffffffeu;
        narrow((uint32_t)kTopkCand, true);
      }
    }
    ties = in_bin > (uint32_t)kTopkCand;
    // ---- 5: keys above the bin are taken; the keys of the bin become candidates (or, all equal and many, a bitmap)
    for (int e = tid; e < n_list && !ranked; e += TH) {
      const uint32_t kk = list_key[e], j = list_idx[e];
      if (kk >= lo) {
        if (kk - lo > span) atomicOr(&take_w[j >> 5], 1u << (j & 31u));
        else if (ties) atomicOr(&eq_w[j >> 5], 1u << (j & 31u));
        else {
          const uint32_t at = atomicAdd(&sh_cand, 1u);
          if (at < (uint32_t)kTopkCand) cand_s[at] = ((unsigned long long)kk << 32) | (0xffffffffu - j);
        }
      }
    }
    __syncthreads();
    in_bin = min(in_bin, sh_cand);                         // what cand_s holds
    if (!ties && (uint32_t)warp < in_bin) {
      constexpr int CL = kTopkCand / 32;
      unsigned long long held[CL];                         // this lane's share of the candidates
#pragma unroll
      for (int i = 0; i < CL; ++i) held[i] = (uint32_t)(lane + 32 * i) < in_bin ? cand_s[lane + 32 * i] : 0ull;
#pragma unroll 2
      for (uint32_t e = (uint32_t)warp; e < in_bin; e += NWARP) {
        const unsigned long long mine = cand_s[e];
        uint32_t before = 0;
#pragma unroll
        for (int i = 0; i < CL; ++i) before += held[i] > mine ? 1u : 0u;
        before = __reduce_add_sync(0xffffffffu, before);
        const uint32_t j = 0xffffffffu - (uint32_t)mine;
        if (lane == 0 && before < need) atomicOr(&take_w[j >> 5], 1u << (j & 31u));
      }
    }
  }
  // Algorithm 2 line 5: the head's static outlier chunks join the set
  if (n_out > 0) {
    const int32_t* outl = outliers + (size_t)prob * (size_t)n_out;     // [G][batch][H_kv][n_out], like sel_idx
    for (int o = tid; o < n_out; o += TH) {
      const int jo = outl[o];
      if (jo >= 0 && jo < n_c) atomicOr(&take_w[jo >> 5], 1u << (jo & 31));
    }
  }
  __syncthreads();
  // ---- 6: exclusive prefix over the CTA in thread order (thread w owns word w), and the total
  auto block_scan = [&](uint32_t mine, uint32_t* tot, uint32_t& total) -> uint32_t {
    uint32_t inc = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t v = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += v;
    }
    if (lane == 31) tot[warp] = inc;
    __syncthreads();
    const uint32_t t = lane < NWARP ? tot[lane] : 0u;
    total = __reduce_add_sync(0xffffffffu, t);
    return inc - mine + __reduce_add_sync(0xffffffffu, lane < warp ? t : 0u);
  };
  uint32_t fw = tid < NW ? take_w[tid] : 0u;
  if (ties) {                                              // of the equal keys, the `need` with the lowest chunk index
    const uint32_t ew = tid < NW ? eq_w[tid] : 0u;
    uint32_t total;
    const uint32_t eq_before = block_scan((uint32_t)__popc(ew), warp_eq, total);
    uint32_t room = need > eq_before ? need - eq_before : 0u;
    uint32_t rest = ew;
    while (rest && room) { fw |= rest & (0u - rest); rest &= rest - 1u; --room; }   // lowest set bits first
  }
  uint32_t taken;
  uint32_t pos = block_scan((uint32_t)__popc(fw), warp_tot, taken);
  // whole chunks unless the ragged last chunk was taken (it is then the last one)
  if (tid == (n_c - 1) >> 5) sh[0] = (fw >> ((n_c - 1) & 31)) & 1u;
  // chunk ids to the chunk list (ascending), rows written by the whole CTA
  for (uint32_t rest = fw; rest; rest &= rest - 1u) list_key[pos++] = (uint32_t)(tid * 32 + __ffs(rest) - 1);
  __syncthreads();
  if (c == 8) {
    for (uint32_t w = (uint32_t)tid; w < taken * 8u; w += TH) {
      const int row = (int)list_key[w >> 3] * 8 + (int)(w & 7u);
      if (row < T) out[w] = row;
    }
  } else {
    for (uint32_t w = (uint32_t)tid; w < taken * (uint32_t)c; w += TH) {
      const uint32_t e = w / (uint32_t)c, t = w - e * (uint32_t)c;
      const int row = (int)list_key[e] * c + (int)t;
      if (row < T) out[w] = row;
    }
  }
  int cnt = (int)taken * c;
  if (sh[0]) cnt -= (n_c * c - T);
  for (int i = cnt + tid; i < k_cap; i += TH) out[i] = -1;
  if (tid == 0 && sel_cnt) sel_cnt[prob] = cnt;
}

}  // namespace

// Top-k of `problems` rows of dev.pooled (sign == 0: keys; else floats compared as sign * value).
static cudaError_t launch_topk(const GroupDev& dev, int device, int problems, int l0, int k_ch, int k_cap,
                               const int32_t* outliers, int n_out, float sign, const __nv_bfloat16* q, int32_t* sel_idx,
                               int32_t* sel_cnt, cudaStream_t s) {   // q: not null if the keys are score_bound_kernel's
  if (dev.n_c > kTopkThreads * 32)
    return launch_pdl(topk_kernel, dim3(problems), dim3(kTopkThreads), 0, s, dev, l0, k_ch, k_cap, outliers, n_out,
                      sign, sel_idx, sel_cnt);
  // keys per thread: 16 up to 16384 chunks, 32 beyond; threads: the fewest of 128, 256, 512, 1024 that cover the
  // chunks (a short context needs fewer barriers' worth of warps, and several of its CTAs share an SM); groups per
  // thread: the fewest with at least k_ch groups in all (0 = no filter)
  int sms = 0;
  cudaError_t e = device_sms(device, &sms);
  if (e != cudaSuccess) return e;
  const int items = dev.n_c <= kTopkThreads * 16 ? 16 : 32;
  auto groups = [&](int gpt) { return (dev.n_c + items / gpt - 1) / (items / gpt); };
  int th = items == 32 ? 1024 : (dev.n_c <= 128 * 16 ? 128 : dev.n_c <= 256 * 16 ? 256 : dev.n_c <= 512 * 16 ? 512 : 1024);
  if (groups(4) < k_ch && th < 512) th *= 2;       // no filter: every key is listed, more threads pay
  // Where a CTA has its SM to itself small ones leave room for nobody.  Selections of 4 to 128 problems, base threads
  // against twice as many: 2048 rows 7.27 -> 7.05 us, 16384 rows and budget 2048 10.6 -> 9.4, 32768 rows 13.3 -> 12.1 (128
  // problems 38.6 -> 38.2); with 256 problems 2048 rows lose (9.0 -> 10.0).  From 512 to 1024 threads the barriers cost
  // more than the threads bring (65536 rows, 8 problems, budget 2048: 8.9 -> 9.7 us), unless the lists are long (4
  // problems, budget 8192: 10.5 -> 10.1) or the problems many (window of 128: 158.2 -> 157.5 us).
  if (q && th < 512) th = 512;                     // (a thread per piece of the queries, a warp per chunk of the band)
  if (problems <= sms && (th < 512 || (th == 512 && (problems > sms / 4 || groups(1) < k_ch)))) th *= 2;
  const size_t smem = (size_t)th * items * (sizeof(uint32_t) + sizeof(uint16_t));
#define XKV_PIVOT(GPT, ITEMS, TH, BOUND)                                                                              \
  do {                                                                                                                \
    e = ensure_dyn_smem<topk_pivot_kernel<GPT, ITEMS, TH, BOUND>>(smem, device);                                      \
    if (e == cudaSuccess)                                                                                             \
      e = launch_pdl(topk_pivot_kernel<GPT, ITEMS, TH, BOUND>, dim3(problems), dim3(TH), smem, s, dev, l0, k_ch, k_cap, \
                     outliers, n_out, sign, q, sel_idx, sel_cnt);                                                     \
  } while (0)
#define XKV_PIVOT_G(ITEMS, TH, BOUND)                                                                                 \
  do {                                                                                                                \
    if (groups(1) >= k_ch) XKV_PIVOT(1, ITEMS, TH, BOUND);                                                            \
    else if (groups(2) >= k_ch) XKV_PIVOT(2, ITEMS, TH, BOUND);                                                       \
    else if (groups(4) >= k_ch) XKV_PIVOT(4, ITEMS, TH, BOUND);                                                       \
    else XKV_PIVOT(0, ITEMS, TH, BOUND);                                                                              \
  } while (0)
  if (q) {
    if (items == 32) XKV_PIVOT_G(32, 1024, true);
    else if (th == 512) XKV_PIVOT_G(16, 512, true);
    else XKV_PIVOT_G(16, 1024, true);
  } else if (items == 32) XKV_PIVOT_G(32, 1024, false);
  else if (th == 128) XKV_PIVOT_G(16, 128, false);
  else if (th == 256) XKV_PIVOT_G(16, 256, false);
  else if (th == 512) XKV_PIVOT_G(16, 512, false);
  else XKV_PIVOT_G(16, 1024, false);
#undef XKV_PIVOT_G
#undef XKV_PIVOT
  return e;
}

// Both kernels of the selection for the problems of layers [l0, l1); `tmap` describes dev.landmarks.
// The caller has checked that the row stride (ceil(k/c) + n_out) * c fits 32 bits (select_stride_ok).
static cudaError_t launch_select_dev(const GroupDev& dev, const CUtensorMap& tmap, int device, int l0, int l1,
                                     const __nv_bfloat16* q, int k, int32_t* sel_idx, int32_t* sel_cnt, cudaStream_t s) {
  const int problems = (l1 - l0) * dev.batch * dev.H_kv;
  const int tiles = (dev.n_c + kScoreRows - 1) / kScoreRows;
  const int c = dev.c;
  const int k_ch_raw = (int)(((int64_t)k + c - 1) / c);
  const int k_ch = k_ch_raw < dev.n_c ? k_ch_raw : dev.n_c;
  const int k_cap = (k_ch_raw + dev.n_out) * c;      // room for the union with the outlier chunks
  dim3 grid(tiles, problems);
  cudaError_t e;
  // Tensor-core scores with a bound pay where the scan is more than a few microseconds of work: the band costs the top-k 1.5
  // to 3 us.  Selections, canonical scan -> bound: 7 heads, 65536 rows, 128 problems 67.3 -> 46.4 us, 64 problems 37.8 -> 26.9,
  // 16 problems 15.7 -> 12.7, 8192 rows and 128 problems 16.5 -> 14.7, 32768 rows and 16 problems 10.2 -> 10.6, 2048 rows and
  // 128 problems 9.7 -> 12.4; 5 heads, 16384 rows, 64 problems 14.4 -> 14.0, 32768 rows and 16 problems 9.3 -> 10.4; 16 heads,
  // 131072 rows, 64 problems 135.8 -> 47.3, 32768 rows and 16 problems 14.9 -> 11.6, 16384 rows and 16 problems 11.9 -> 12.0.
  // Without a handle there is no room for the tiles' sums.
  const bool bound = dev.tile_sum != nullptr && dev.n_rep > 4 && k_ch < dev.n_c && dev.n_c <= kTopkThreads * 32 &&
                     (int64_t)problems * dev.n_c * dev.n_rep >= 5 << 17;
  const size_t smem = 1024 + (size_t)(dev.d_h / 64) * kScoreRows * 128 + (bound ? 0 : (size_t)dev.n_rep * dev.d_h * 4);
#define XKV_SCAN_BOUND(DH, NT)                                                                          \
  do {                                                                                                  \
    e = ensure_dyn_smem<score_bound_kernel<DH, NT>>(smem, device);                                      \
    if (e != cudaSuccess) return e;                                                                     \
    e = launch_pdl(score_bound_kernel<DH, NT>, grid, dim3(kScoreThreads), smem, s, tmap, dev, q, l0);   \
  } while (0)
#define XKV_SCAN(DH, HMAX)                                                                              \
  do {                                                                                                  \
    e = ensure_dyn_smem<score_pool_kernel<DH, HMAX>>(smem, device);                                     \
    if (e != cudaSuccess) return e;                                                                     \
    e = launch_pdl(score_pool_kernel<DH, HMAX>, grid, dim3(kScoreThreads), smem, s, tmap, dev, q, l0); \
  } while (0)
  if (bound) {
    if (dev.d_h == 128) { if (dev.n_rep <= 8) XKV_SCAN_BOUND(128, 1); else XKV_SCAN_BOUND(128, 2); }
    else { if (dev.n_rep <= 8) XKV_SCAN_BOUND(64, 1); else XKV_SCAN_BOUND(64, 2); }
  } else if (dev.d_h == 128) {
    if (dev.n_rep <= 4) XKV_SCAN(128, 4); else XKV_SCAN(128, 8);
  } else {
    if (dev.n_rep <= 4) XKV_SCAN(64, 4); else XKV_SCAN(64, 8);
  }
#undef XKV_SCAN
#undef XKV_SCAN_BOUND
  count_launch(kFamScan);
  if (e != cudaSuccess) return e;
  e = launch_topk(dev, device, problems, l0, k_ch, k_cap, dev.outliers, dev.n_out, 0.0f, bound ? q : nullptr, sel_idx, sel_cnt, s);
  count_launch(kFamTopk);
  return e;
}

// (ceil(k/c) + n_out) * c, the row stride of sel_idx, must fit the 32-bit arithmetic of the kernels.
bool select_stride_ok(int64_t k, int c, int n_out) {
  return k >= 1 && ((k + c - 1) / c + n_out) * (int64_t)c < ((int64_t)1 << 30);
}

// The k entries with the largest sign * scores[p][j] of each of `problems` score rows of length n, ids ascending
// (ties to the lowest id), padded with -1: out [problems][k].  Used for the static outlier chunks (Algorithm 1 line 5).
cudaError_t launch_topk_rows(const float* scores, int problems, int n, int k, float sign, int32_t* out, int device,
                             cudaStream_t s) {
  GroupDev dev{};
  dev.G = 1; dev.batch = problems; dev.H_kv = 1; dev.T = n; dev.c = 1; dev.n_c = n;
  dev.pooled = const_cast<float*>(scores);
  const int k_ch = k < n ? k : n;
  cudaError_t e = launch_topk(dev, device, problems, 0, k_ch, k, nullptr, 0, sign, nullptr, out, nullptr, s);
  count_launch(kFamTopk);
  return e;
}

cudaError_t launch_select(const xkv_group* grp, int l0, int l1, const __nv_bfloat16* q, int k,
                          int32_t* sel_idx, int32_t* sel_cnt, cudaStream_t s) {
  CUtensorMap tmap;
  memcpy(&tmap, grp->lm_tmap, sizeof(tmap));
  return launch_select_dev(grp->dev, tmap, grp->device, l0, l1, q, k, sel_idx, sel_cnt, s);
}

// ---------------------------------------------------------------------------------------------
// Selection without a handle and without any allocation: the pooled scores live in a file-scope device array.

// 64 flag words followed by the pooled scores of every problem of the call.
static __device__ __align__(256) float g_static_scratch[64 + XKV_STATIC_SELECT_MAX_SCORES];

// The array's name is only a host-side stand-in; its device address is looked up once per device.
static float* static_scratch_ptr(int device, cudaError_t* err) {
  static std::mutex mu;
  static float* ptrs[64] = {};
  std::lock_guard<std::mutex> lock(mu);
  *err = cudaSuccess;
  if (device < 0 || device >= 64) { *err = cudaErrorInvalidDevice; return nullptr; }
  if (!ptrs[device]) {
    float* p = nullptr;
    *err = cudaGetSymbolAddress((void**)&p, g_static_scratch);   // the current device is `device`
    if (*err != cudaSuccess) return nullptr;
    ptrs[device] = p;
  }
  return ptrs[device];
}

int select_static(const xkv_select_static_config* c, int l0, int l1, const void* q, int32_t k, int32_t* sel_idx,
                  int32_t* sel_cnt, cudaStream_t s) {
  if (!c || !q || !sel_idx || !sel_cnt || c->struct_size != sizeof(xkv_select_static_config)) return XKV_ERR_INVALID_ARG;
  if (c->G < 1 || c->batch < 1 || c->T < 1 || c->T >= (1 << 24) || c->H_kv < 1 || c->H_q < 1 ||
      c->H_q % c->H_kv != 0 || c->H_q / c->H_kv > kMaxRep || (c->d_h != 64 && c->d_h != 128) || c->chunk < 0 ||
      c->chunk > 4096 || !c->landmarks || ((uintptr_t)c->landmarks & 15u) || ((uintptr_t)q & 15u) ||
      ((uintptr_t)sel_idx & 3u) || ((uintptr_t)sel_cnt & 3u))
    return XKV_ERR_INVALID_ARG;
  if (l0 < 0 || l1 > c->G || l0 >= l1 || k < 1) return XKV_ERR_INVALID_ARG;
  // a budget beyond the context means "every row"; the row stride the caller allocated follows from k, so a k whose
  // stride leaves 32-bit range is rejected here, before anything is launched
  if (!select_stride_ok(k, c->chunk ? c->chunk : 8, 0)) return XKV_ERR_INVALID_ARG;
  GroupDev dev{};
  dev.G = c->G; dev.batch = c->batch; dev.T = c->T; dev.H_kv = c->H_kv; dev.H_q = c->H_q; dev.d_h = c->d_h;
  dev.c = c->chunk ? c->chunk : 8;
  dev.n_c = (c->T + dev.c - 1) / dev.c;
  dev.n_rep = c->H_q / c->H_kv;
  dev.sel_scale = 1.0f / sqrtf((float)c->d_h);
  dev.landmarks = (const __nv_bfloat16*)c->landmarks;
  const size_t scores = (size_t)c->G * c->batch * c->H_kv * dev.n_c;   // indexed by absolute layer, like the handle's
  if (scores > (size_t)XKV_STATIC_SELECT_MAX_SCORES) return XKV_ERR_TOO_LARGE;
  if ((size_t)c->G * c->batch * c->H_kv > 65535) return XKV_ERR_TOO_LARGE;   // problems of a call are a grid dimension
  int device = 0;
  cudaError_t e = cudaGetDevice(&device);
  if (e != cudaSuccess) { set_cuda_error(e); return XKV_ERR_CUDA; }
  static std::atomic<int> cc_major[kMaxDevices];          // 0: not looked up yet
  if (device < 0 || device >= kMaxDevices) return XKV_ERR_ARCH;
  int major = cc_major[device].load(std::memory_order_relaxed);
  if (major == 0) {
    e = cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, device);
    if (e != cudaSuccess) { set_cuda_error(e); return XKV_ERR_CUDA; }
    cc_major[device].store(major, std::memory_order_relaxed);
  }
  if (major != 10) return XKV_ERR_ARCH;
  float* scratch = static_scratch_ptr(device, &e);
  if (!scratch) { set_cuda_error(e); (void)cudaGetLastError(); return XKV_ERR_CUDA; }
  dev.flags = reinterpret_cast<unsigned int*>(scratch);
  dev.pooled = scratch + 64;
  CUtensorMap tmap;
  if (!encode_landmark_map(&tmap, c->landmarks, (uint64_t)c->batch * c->G * c->H_kv * dev.n_c, (uint64_t)c->d_h))
    return XKV_ERR_CUDA;
  e = cudaMemsetAsync(scratch, 0, 64 * sizeof(float), s);              // the flag words start at zero
  if (e == cudaSuccess) e = launch_select_dev(dev, tmap, device, l0, l1, (const __nv_bfloat16*)q, k, sel_idx, sel_cnt, s);
  if (e != cudaSuccess) { set_cuda_error(e); (void)cudaGetLastError(); return XKV_ERR_CUDA; }
  return XKV_OK;
}

}  // namespace xkv
