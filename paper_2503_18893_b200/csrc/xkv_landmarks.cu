// Landmark construction at prefill (App. B.1, Algorithm 1): chunk means of the post-RoPE keys and, optionally, the
// minimum within-chunk cosine similarity to the chunk mean, from which the static outlier chunks are taken.
// HBM bound: every key row is read once from DRAM (a second time from cache when the cosines are wanted, because
// they need the finished mean).
// One CTA handles up to 32 consecutive rows (whole chunks when c <= 32) of one (sequence, layer) for all KV heads.
// A thread owns 8 rotary pairs of one head (16-byte loads of the two halves of the row) and walks the rows of a
// chunk; the CTA's row groups work on different chunks.  The cos/sin of p * theta_i are formed in fp64 for the
// first row of the CTA (the angle reaches 2^24 rad; sincospi reduces it exactly) and advanced row by row with the
// fp64 rotation by theta_i; all heads share them through shared memory.
#include <math.h>

#include "xkv_internal.cuh"
#include "xkv_ptx.cuh"

namespace xkv {

namespace {

constexpr int kLmRows = 32;         // key rows per table (per CTA pass)
constexpr int kLmThreads = 256;

__device__ __forceinline__ void unpack8(const uint4& v, float (&f)[8]) {
  const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
  for (int e = 0; e < 4; ++e) { f[2 * e] = __uint_as_float(w[e] << 16); f[2 * e + 1] = __uint_as_float(w[e] & 0xffff0000u); }
}
__device__ __forceinline__ uint4 pack8(const float (&f)[8]) {
  uint4 v;
  __nv_bfloat162 t;
  t = __floats2bfloat162_rn(f[0], f[1]); v.x = *reinterpret_cast<uint32_t*>(&t);
  t = __floats2bfloat162_rn(f[2], f[3]); v.y = *reinterpret_cast<uint32_t*>(&t);
  t = __floats2bfloat162_rn(f[4], f[5]); v.z = *reinterpret_cast<uint32_t*>(&t);
  t = __floats2bfloat162_rn(f[6], f[7]); v.w = *reinterpret_cast<uint32_t*>(&t);
  return v;
}

// keys      bf16 [batch][G][T][H_kv*d_h], rows before rotation (use_rope) or already rotated
// landmarks bf16 [batch][G][H_kv][n_c][d_h]
// min_cos   fp32 [G][batch][H_kv][n_c] or nullptr
// grid = (ceil(n_c / chunks per CTA), G, batch), block = kLmThreads.  TPR = H_kv * d_h / 16 threads cover one row;
// TPR divides kLmThreads (checked on the host); the 8 or 4 threads of a head are consecutive lanes of one warp.
template <int DH>
__global__ void __launch_bounds__(kLmThreads, 3)
landmark_kernel(const __nv_bfloat16* __restrict__ keys, __nv_bfloat16* __restrict__ landmarks, float* __restrict__ min_cos,
                int G, int batch, int T, int H_kv, int c, int n_c, int chunks_per_cta, double rope_base, int use_rope) {
  constexpr int HALF = DH / 2;
  constexpr int APH = HALF / 8;                          // threads per head: each owns 8 rotary pairs
  __shared__ __align__(16) float2 cs_s[kLmRows * HALF];  // (cos, sin) of (row, pair) for the rows of the current pass
  __shared__ float comb_s[kLmThreads][17];               // long chunks only: partial results of the row groups
  const int tid = threadIdx.x;
  const int TPR = H_kv * APH, RG = kLmThreads / TPR;     // threads per row, row groups
  const int rg = tid / TPR, tr = tid % TPR;
  const int g = tr / APH, a = tr % APH;
  const int l = blockIdx.y, b = blockIdx.z;
  const int d = H_kv * DH;
  const __nv_bfloat16* K = keys + (((size_t)b * G + l) * T) * d + (size_t)g * DH + a * 8;
  const bool whole = c <= kLmRows;                        // all chunks of this CTA share one table
  const int R0 = blockIdx.x * chunks_per_cta * c;

  // cos/sin of rows [first, first + n): thread -> (pair, block of consecutive rows); the block's first row by
  // sincospi, then one fp64 rotation by theta per row
  auto fill_table = [&](int first, int n) {
    constexpr int BLKS = kLmThreads / HALF, RPB = kLmRows / BLKS;   // 4 blocks of 8 rows (d_h = 128), 8 of 4 (d_h = 64)
    const int ii = tid % HALF, r_begin = (tid / HALF) * RPB;
    if (r_begin < n) {
      const double th = pow(rope_base, -(double)ii / (double)HALF);
      double sn, cs, st, ct;
      sincospi((double)(first + r_begin) * (th / 3.14159265358979323846), &sn, &cs);
      sincos(th, &st, &ct);                               // theta <= 1: no range reduction needed
      const int r_end = min(n, r_begin + RPB);
      for (int r = r_begin; r < r_end; ++r) {
        cs_s[r * HALF + ii] = make_float2((float)cs, (float)sn);
        const double c2 = cs * ct - sn * st, s2 = sn * ct + cs * st;
        cs = c2; sn = s2;
      }
    }
  };
  // one row: this thread's 8 pairs -> x1[8] (dims a*8..), x2[8] (dims HALF + a*8..), rotated with table row `trow`
  auto load_row = [&](int row, uint4& u1, uint4& u2) {
    const __nv_bfloat16* kr = K + (size_t)row * d;
    u1 = __ldg(reinterpret_cast<const uint4*>(kr));
    u2 = __ldg(reinterpret_cast<const uint4*>(kr + HALF));
  };
  auto rotate = [&](const uint4& u1, const uint4& u2, int trow, float (&x1)[8], float (&x2)[8]) {
    unpack8(u1, x1); unpack8(u2, x2);
    if (use_rope) {
      const float4* t4 = reinterpret_cast<const float4*>(cs_s + trow * HALF + a * 8);
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const float4 t = t4[e];                           // (cos, sin) of pairs 2e and 2e+1
        const float y1 = x1[2 * e] * t.x - x2[2 * e] * t.y, y2 = x2[2 * e] * t.x + x1[2 * e] * t.y;
        const float z1 = x1[2 * e + 1] * t.z - x2[2 * e + 1] * t.w, z2 = x2[2 * e + 1] * t.z + x1[2 * e + 1] * t.w;
        x1[2 * e] = y1; x2[2 * e] = y2; x1[2 * e + 1] = z1; x2[2 * e + 1] = z2;
      }
    }
  };
  // sum over the APH threads of a head (consecutive lanes)
  // (only those lanes take part: the row groups of a warp may be in different chunks)
  const uint32_t hmask = ((1u << APH) - 1u) << ((tid & 31) & ~(APH - 1));
  auto head_sum = [&](float v) {
#pragma unroll
    for (int o = 1; o < APH; o <<= 1) v += __shfl_xor_sync(hmask, v, o);
    return v;
  };
  auto cosine = [&](const float (&x1)[8], const float (&x2)[8], const float (&m1)[8], const float (&m2)[8], float mn2) {
    float dot = 0.0f, nn = 0.0f;
#pragma unroll
    for (int e = 0; e < 8; ++e) { dot += x1[e] * m1[e] + x2[e] * m2[e]; nn += x1[e] * x1[e] + x2[e] * x2[e]; }
    dot = head_sum(dot); nn = head_sum(nn);
    const float den = sqrtf(nn) * sqrtf(mn2);
    return den > 0.0f ? dot / den : 0.0f;
  };

  if (whole) {
    if (use_rope) {
      fill_table(R0, min(chunks_per_cta * c, T - R0));
      __syncthreads();
    }
    // ---- chunks of at most 32 rows: row group rg takes chunks rg, rg + RG, ... of this CTA
    for (int jc = rg; jc < chunks_per_cta; jc += RG) {
      const int j = blockIdx.x * chunks_per_cta + jc;
      if (j >= n_c) break;
      const int row0 = j * c, rows = min(c, T - row0);
      float m1[8], m2[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) { m1[e] = 0.0f; m2[e] = 0.0f; }
      for (int rb = 0; rb < rows; rb += 4) {              // four rows' loads in flight
        uint4 u1[4], u2[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) load_row(row0 + min(rb + u, rows - 1), u1[u], u2[u]);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          if (rb + u < rows) {
            float x1[8], x2[8];
            rotate(u1[u], u2[u], row0 - R0 + rb + u, x1, x2);
#pragma unroll
            for (int e = 0; e < 8; ++e) { m1[e] += x1[e]; m2[e] += x2[e]; }
          }
        }
      }
      const float inv = 1.0f / (float)rows;
#pragma unroll
      for (int e = 0; e < 8; ++e) { m1[e] *= inv; m2[e] *= inv; }
      __nv_bfloat16* L = landmarks + ((((size_t)b * G + l) * H_kv + g) * n_c + j) * DH + a * 8;
      *reinterpret_cast<uint4*>(L) = pack8(m1);
      *reinterpret_cast<uint4*>(L + HALF) = pack8(m2);
      if (min_cos) {
        float mn2 = 0.0f;
#pragma unroll
        for (int e = 0; e < 8; ++e) mn2 += m1[e] * m1[e] + m2[e] * m2[e];
        mn2 = head_sum(mn2);
        float best = INFINITY;
        for (int rb = 0; rb < rows; rb += 4) {
          uint4 u1[4], u2[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) load_row(row0 + min(rb + u, rows - 1), u1[u], u2[u]);
#pragma unroll
          for (int u = 0; u < 4; ++u) {                    // a repeated last row changes no minimum
            float x1[8], x2[8];
            rotate(u1[u], u2[u], row0 - R0 + min(rb + u, rows - 1), x1, x2);
            best = fminf(best, cosine(x1, x2, m1, m2, mn2));
          }
        }
        if (a == 0) min_cos[(((size_t)l * batch + b) * H_kv + g) * n_c + j] = best;
      }
    }
    return;
  }

  // ---- a chunk longer than 32 rows: one chunk per CTA, passes of 32 rows, the row groups split the rows of a pass
  const int j = blockIdx.x;
  const int row0 = j * c, rows = min(c, T - row0);
  float m1[8], m2[8];
#pragma unroll
  for (int e = 0; e < 8; ++e) { m1[e] = 0.0f; m2[e] = 0.0f; }
  float mn2 = 0.0f, best = INFINITY;
  for (int phase = 0; phase < (min_cos ? 2 : 1); ++phase) {
    for (int r0 = 0; r0 < rows; r0 += kLmRows) {
      const int nr = min(kLmRows, rows - r0);
      __syncthreads();                                    // the previous pass is done with the table
      if (use_rope) fill_table(row0 + r0, nr);
      __syncthreads();
      for (int r = rg; r < nr; r += RG) {
        uint4 u1, u2;
        load_row(row0 + r0 + r, u1, u2);
        float x1[8], x2[8];
        rotate(u1, u2, r, x1, x2);
        if (phase == 0) {
#pragma unroll
          for (int e = 0; e < 8; ++e) { m1[e] += x1[e]; m2[e] += x2[e]; }
        } else {
          best = fminf(best, cosine(x1, x2, m1, m2, mn2));
        }
      }
    }
    // combine the row groups: sums (phase 0) or minima (phase 1) of the same (head, pair group)
    __syncthreads();
    if (phase == 0) {
#pragma unroll
      for (int e = 0; e < 8; ++e) { comb_s[tid][e] = m1[e]; comb_s[tid][8 + e] = m2[e]; }
      __syncthreads();
#pragma unroll
      for (int e = 0; e < 8; ++e) { m1[e] = 0.0f; m2[e] = 0.0f; }
      for (int q = 0; q < RG; ++q) {
#pragma unroll
        for (int e = 0; e < 8; ++e) { m1[e] += comb_s[q * TPR + tr][e]; m2[e] += comb_s[q * TPR + tr][8 + e]; }
      }
      const float inv = 1.0f / (float)rows;
#pragma unroll
      for (int e = 0; e < 8; ++e) { m1[e] *= inv; m2[e] *= inv; }
      if (rg == 0) {
        __nv_bfloat16* L = landmarks + ((((size_t)b * G + l) * H_kv + g) * n_c + j) * DH + a * 8;
        *reinterpret_cast<uint4*>(L) = pack8(m1);
        *reinterpret_cast<uint4*>(L + HALF) = pack8(m2);
      }
#pragma unroll
      for (int e = 0; e < 8; ++e) mn2 += m1[e] * m1[e] + m2[e] * m2[e];
      mn2 = head_sum(mn2);
    } else {
      comb_s[tid][16] = best;
      __syncthreads();
      for (int q = 0; q < RG; ++q) best = fminf(best, comb_s[q * TPR + tr][16]);
      if (rg == 0 && a == 0) min_cos[(((size_t)l * batch + b) * H_kv + g) * n_c + j] = best;
    }
  }
}

using namespace ptx;                // packed fp32

// The default chunk of 8 rows (c == 8), persistent CTAs.  The arithmetic of the kernel above, landmarks operation by
// operation; two things may move a last bit.  The table entries come from an fp64 rotation carried from block to block
// instead of a sincospi per 4 or 8 rows (apart by the rounding of an fp64 angle; as fp32 they differ so rarely that 7 of
// 512 M landmark elements do at 1000003 rows of 32 heads, none at 131072 rows of four layers of 8), and the sums of a cosine over the lanes
// of a head are folded in another order (1e-5 of the cosines, by 1.2e-7).  The error against fp64 is that of the kernel
// above: cosines 2.4e-7 at most, 5.7e-8 rms; 261 of 8.4 M landmarks on the other side of a rounding boundary, for both.
// A CTA walks a contiguous range of row blocks; the cos/sin table of a block is built once and serves every (sequence,
// layer) and head, so its fp64 work (an eighth of the fp32 rate here) is divided by batch * G: per CTA and layer, as in
// the kernel above, it took as long as everything else together.  The rotation is advanced in fp64 from block to block;
// pow and sincos run once per CTA.
// A thread holds the 8 rows of its 8 rotary pairs in registers, so nothing is read again, while its next chunks are on the
// way into 256 bytes each of shared memory of its own (no barrier: nobody else reads them).  The arithmetic is packed fp32
// (two pairs per instruction), the sums of the cosine pass over the threads of a head are folded by halving (a lane ends
// with one row: 14 shuffles for the 16 sums of a chunk instead of 6 per row).
// With cosines the rotated rows stay in registers too (128 of them): a 16-byte load for every thread of a warp takes the
// shared-memory pipe four cycles whether the addresses agree or not, and the second reading of the table, with the second
// rotation, was a third of the instructions and of that pipe's time.  That leaves room for one CTA per SM, which keeps two
// chunks per thread on their way.  131072 rows of four layers of eight heads of 128: 296 us with two CTAs rotating twice,
// 239 with one (5.1 TB/s); 2048 rows 21.4 -> 16.4.  Without cosines two CTAs per SM with the raw rows in registers: 211 us
// (5.7 TB/s; 197 without rotation).  What is left is the start of a CTA (pow, sincospi) and 64 to 128 KB in flight per SM.
constexpr int kLm8MaxRows = 64;     // rows of a table
template <int DH, bool ROPE, bool COS>
__global__ void __launch_bounds__(kLmThreads, COS ? 1 : 2)
landmark8_kernel(const __nv_bfloat16* __restrict__ keys, __nv_bfloat16* __restrict__ landmarks, float* __restrict__ min_cos,
                 int G, int batch, int T, int H_kv, int n_c, int CPB, int n_blocks, int two_tables, double rope_base) {
  constexpr int HALF = DH / 2, APH = HALF / 8, NBLK = kLmThreads / HALF;
  constexpr int SLOTS = COS ? 2 : 1;                     // chunks of a thread on their way
  extern __shared__ __align__(16) uint4 slots_s[];       // [SLOTS][16][kLmThreads] pieces of the chunks on their way, then the tables
  __shared__ double2 rot_s[3][ROPE ? kLmThreads : 1];    // a thread's rotation state: its first row, one row on, one block on
  const int tid = threadIdx.x;
  const int TPR = H_kv * APH, RG = kLmThreads / TPR;     // threads per row of all heads, chunks side by side
  const int R = CPB * 8, LG = RG / CPB;                  // rows of a block; beyond CPB chunks the row groups take other layers
  const int rg = tid / TPR, tr = tid % TPR;
  const int g = tr / APH, a = tr % APH;
  const int jc = rg % CPB, lg = rg / CPB;
  const int d = H_kv * DH, n_lb = G * batch;
  const int b_begin = (int)((long long)blockIdx.x * n_blocks / gridDim.x), b_end = (int)((long long)(blockIdx.x + 1) * n_blocks / gridDim.x);
  float4* const tab_s = reinterpret_cast<float4*>(slots_s + SLOTS * 16 * kLmThreads);     // [row][4][APH] {cos, cos, sin, sin} of two pairs

  // this thread's share of the table: pair ii, rows [r_begin, r_begin + RPB) of every block
  const int ii = tid % HALF, RPB = max(1, R / NBLK), r_begin = (tid / HALF) * RPB;
  const bool fills = r_begin < R;
  if (ROPE && fills) {
    const double th = pow(rope_base, -(double)ii / (double)HALF);
    double2 v;
    sincospi((double)(b_begin * R + r_begin) * (th / 3.14159265358979323846), &v.y, &v.x);
    rot_s[0][tid] = v;
    sincos(th, &v.y, &v.x);                               // theta <= 1: no range reduction needed
    rot_s[1][tid] = v;
    sincospi((double)R * (th / 3.14159265358979323846), &v.y, &v.x);
    rot_s[2][tid] = v;
  }
  float* const tab_f = reinterpret_cast<float*>(tab_s) + ((((ii & 7) >> 1) * APH + (ii >> 3)) * 4 + (ii & 1));
  const ulonglong2* const tab0 = reinterpret_cast<const ulonglong2*>(tab_s) + a;
  const int tab_floats = R * HALF * 2;                    // of one table

  uint4 u1[8], u2[8];
  const uint32_t slot_addr = ptx::smem_u32(slots_s + tid);
  auto request_chunk = [&](int blk, int lb, int at) {     // lb = sequence * G + layer
    const int j = blk * CPB + jc;
    if (blk >= b_end || j >= n_c || lb >= n_lb) return;
    const int row0 = j * 8, last = min(8, T - row0) - 1;
    const __nv_bfloat16* p = keys + ((size_t)lb * T + row0) * d + (size_t)g * DH + a * 8;
    uint32_t to = slot_addr + (uint32_t)at * (16 * kLmThreads * 16);
    auto row = [&]() {
      ptx::cp_async16(to, p, 16u);
      ptx::cp_async16(to + kLmThreads * 16, p + HALF, 16u);
      to += 2 * kLmThreads * 16;
    };
    if (last == 7) {                                      // every chunk but a ragged last one: a row is one addition away
#pragma unroll
      for (int r = 0; r < 8; ++r, p += d) row();
    } else {
#pragma unroll 1
      for (int r = 0; r < 8; ++r) { row(); if (r < last) p += d; }
    }
  };
  // (only the lanes of one head take part: the row groups of a warp may be in different chunks)
  const uint32_t hmask = ((1u << APH) - 1u) << ((tid & 31) & ~(APH - 1));
  // couple e (pairs 2e, 2e + 1) of row r: first half x1, second half x2
  auto couple = [&](int r, int e, u64& x1, u64& x2) {
    const uint32_t w1 = e == 0 ? u1[r].x : e == 1 ? u1[r].y : e == 2 ? u1[r].z : u1[r].w;
    const uint32_t w2 = e == 0 ? u2[r].x : e == 1 ? u2[r].y : e == 2 ? u2[r].z : u2[r].w;
    x1 = pack2(__uint_as_float(w1 << 16), __uint_as_float(w1 & 0xffff0000u));
    x2 = pack2(__uint_as_float(w2 << 16), __uint_as_float(w2 & 0xffff0000u));
  };
  // ca - sb with the product sb rounded first (the scalar instruction negates an operand for nothing, the packed one does not)
  auto fms = [&](u64 c, u64 a, u64 sb) {
    const float2 cf = unpack2(c), af = unpack2(a), bf = unpack2(sb);
    return pack2(fmaf(cf.x, af.x, -bf.x), fmaf(cf.y, af.y, -bf.y));
  };
  auto fill_table = [&](int buf) {                        // the next block's table, and the state one block on
    float* to = tab_f + buf * tab_floats;
    const double2 at = rot_s[0][tid], one = rot_s[1][tid], jump = rot_s[2][tid];
    double c1 = at.x, s1 = at.y;
    for (int r = r_begin; r < r_begin + RPB; ++r) {
      to[(size_t)r * HALF * 2] = (float)c1;
      to[(size_t)r * HALF * 2 + 2] = (float)s1;
      const double c2 = c1 * one.x - s1 * one.y, s2 = s1 * one.x + c1 * one.y;
      c1 = c2; s1 = s2;
    }
    rot_s[0][tid] = make_double2(at.x * jump.x - at.y * jump.y, at.y * jump.x + at.x * jump.y);
  };

  // the chunk that is requested next: this thread's layers of a block, then the next block
  int req_blk = b_begin, req_lb = lg, slot = 0;
  auto request_next = [&](int at) {
    request_chunk(req_blk, req_lb, at);
    asm volatile("cp.async.commit_group;" ::: "memory");
    req_lb += LG;
    if (req_lb >= n_lb) { req_lb = lg; ++req_blk; }
  };
#pragma unroll
  for (int i = 0; i < SLOTS; ++i) request_next(i);
  for (int blk = b_begin; blk < b_end; ++blk) {
    const int buf = two_tables ? (blk - b_begin) & 1 : 0;
    if (ROPE) {
      // With two tables the next block's is written while this one's rows are read: one barrier a block.
      if (!two_tables || blk == b_begin) {
        __syncthreads();                                  // everybody is done with the table of the previous block
        if (fills) fill_table(0);
      }
      __syncthreads();
      if (two_tables && fills && blk + 1 < b_end) fill_table(buf ^ 1);
    }
    const ulonglong2* const tab = tab0 + buf * (tab_floats / 4);
    const int j = blk * CPB + jc;
    for (int lb = lg; lb < n_lb; lb += LG) {
      // this thread's own copies have landed; into registers, and the next chunk on its way
      asm volatile("cp.async.wait_group %0;" ::"n"(SLOTS - 1) : "memory");
      const uint4* const from = slots_s + slot * (16 * kLmThreads) + tid;
#pragma unroll
      for (int r = 0; r < 8; ++r) { u1[r] = from[(2 * r) * kLmThreads]; u2[r] = from[(2 * r + 1) * kLmThreads]; }
      request_next(slot);
      if (SLOTS == 2) slot ^= 1;
      if (j >= n_c) continue;
      const int rows = min(8, T - j * 8);
      u64 s1[4], s2[4];
      u64 y1[COS ? 8 : 1][4], y2[COS ? 8 : 1][4];         // the rotated rows
#pragma unroll
      for (int e = 0; e < 4; ++e) s1[e] = s2[e] = 0ull;
#pragma unroll
      for (int r = 0; r < 8; ++r) {
        if (COS || r < rows) {
          const int trow = jc * 8 + min(r, rows - 1), k = COS ? r : 0;
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            couple(r, e, y1[k][e], y2[k][e]);
            if (ROPE) {
              const ulonglong2 t = tab[((size_t)trow * 4 + e) * APH];
              const u64 x1 = y1[k][e], x2 = y2[k][e];
              y1[k][e] = fms(x1, t.x, mul2(x2, t.y));
              y2[k][e] = fma2(x2, t.x, mul2(x1, t.y));
            }
            if (r < rows) {
              s1[e] = add2(s1[e], y1[k][e]);
              s2[e] = add2(s2[e], y2[k][e]);
            }
          }
        }
      }
      const float inv = 1.0f / (float)rows;
      const u64 inv2 = pack2(inv, inv);
      float m1[8], m2[8];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        s1[e] = mul2(s1[e], inv2);
        s2[e] = mul2(s2[e], inv2);
        const float2 p = unpack2(s1[e]), q = unpack2(s2[e]);
        m1[2 * e] = p.x; m1[2 * e + 1] = p.y; m2[2 * e] = q.x; m2[2 * e + 1] = q.y;
      }
      __nv_bfloat16* L = landmarks + (((size_t)lb * H_kv + g) * n_c + j) * DH + a * 8;
      *reinterpret_cast<uint4*>(L) = pack8(m1);
      *reinterpret_cast<uint4*>(L + HALF) = pack8(m2);
      if constexpr (COS) {
        float v[8], mn2 = 0.0f;                           // per row: dot product with the mean, squared norm
#pragma unroll
        for (int e = 0; e < 8; ++e) mn2 += m1[e] * m1[e] + m2[e] * m2[e];
#pragma unroll
        for (int o = 1; o < APH; o <<= 1) mn2 += __shfl_xor_sync(hmask, mn2, o);
        auto row_sums = [&](int r, float& dot, float& nn) {
          u64 dot2 = 0ull, nn2 = 0ull;                    // (a repeated last row changes no minimum)
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            dot2 = fma2(y2[r][e], s2[e], fma2(y1[r][e], s1[e], dot2));
            nn2 = fma2(y2[r][e], y2[r][e], fma2(y1[r][e], y1[r][e], nn2));
          }
          const float2 p = unpack2(dot2), q = unpack2(nn2);
          dot = p.x + p.y; nn = q.x + q.y;
        };
        // fold by halving: after the step with distance o a lane keeps the half of the rows its bit selects
        auto folded = [&](int o, float lo, float hi) {
          const bool up = (a & o) != 0;
          const float mine = up ? hi : lo, other = up ? lo : hi;
          return mine + __shfl_xor_sync(hmask, other, o);
        };
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          float dot, nn, dot4, nn4;
          row_sums(r, dot, nn);
          row_sums(r + 4, dot4, nn4);
          v[2 * r] = folded(1, dot, dot4); v[2 * r + 1] = folded(1, nn, nn4);
        }
#pragma unroll
        for (int o = 2, n = 4; o < APH; o <<= 1, n >>= 1) {
#pragma unroll
          for (int i = 0; i < n; ++i) v[i] = folded(o, v[i], v[n + i]);
        }
        float best = INFINITY;
#pragma unroll
        for (int i = 0; i < 16 / APH; i += 2) {
          const float den = sqrtf(v[i + 1]) * sqrtf(mn2);
          best = fminf(best, den > 0.0f ? v[i] / den : 0.0f);
        }
#pragma unroll
        for (int o = 1; o < APH; o <<= 1) best = fminf(best, __shfl_xor_sync(hmask, best, o));
        const int b = lb / G, l = lb - b * G;
        if (a == 0) min_cos[(((size_t)l * batch + b) * H_kv + g) * n_c + j] = best;
      }
    }
  }
}

template <int DH>
cudaError_t launch_landmark8(const __nv_bfloat16* keys, __nv_bfloat16* landmarks, float* min_cos, int G, int batch, int T,
                             int H_kv, float rope_base, cudaStream_t s) {
  const int n_c = (T + 7) / 8, tpr = H_kv * DH / 16;
  const int rg = kLmThreads / tpr;
  const bool rope = rope_base > 0.0f, cosines = min_cos != nullptr;
  int cpb = rg < kLm8MaxRows / 8 ? rg : kLm8MaxRows / 8;
  // Two tables, so that a block costs one barrier and its fp64 work runs beside the others' rows (40003 rows of four layers
  // of four heads, without cosines, 57.3 -> 50.5 us).  One CTA of an SM has room for any two, two CTAs for 16 KB tables: 64
  // rows of 32 pairs or 32 rows of 64.  Of 64 pairs the block keeps 64 rows (and one table) only where the row groups
  // beyond 32 rows would find no layer of their own.
  if (DH == 128 && cpb == 8 && !cosines && rg / 4 <= G * batch) cpb = 4;
  const size_t table = rope ? (size_t)cpb * 8 * (DH / 2) * sizeof(float2) : 0;
  const int two_tables = cosines || table <= 16384 ? 1 : 0;
  const int n_blocks = (n_c + cpb - 1) / cpb;
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = device_sms(dev, &sms);
  if (e != cudaSuccess) return e;
  const int ctas = cosines ? sms : 2 * sms;                           // one wave
  const int grid = n_blocks < ctas ? n_blocks : ctas;
  const size_t smem = (size_t)kLmThreads * 256 * (cosines ? 2 : 1) + (two_tables ? 2 : 1) * table;
  const int variant = (rope ? 2 : 0) + (cosines ? 1 : 0);
  auto launch = [&](auto kernel) {
    kernel<<<grid, kLmThreads, smem, s>>>(keys, landmarks, min_cos, G, batch, T, H_kv, n_c, cpb, n_blocks, two_tables,
                                          rope ? (double)rope_base : 1.0);
  };
  if (variant == 3 && (e = ensure_dyn_smem<landmark8_kernel<DH, true, true>>(smem, dev)) == cudaSuccess) launch(landmark8_kernel<DH, true, true>);
  if (variant == 2 && (e = ensure_dyn_smem<landmark8_kernel<DH, true, false>>(smem, dev)) == cudaSuccess) launch(landmark8_kernel<DH, true, false>);
  if (variant == 1 && (e = ensure_dyn_smem<landmark8_kernel<DH, false, true>>(smem, dev)) == cudaSuccess) launch(landmark8_kernel<DH, false, true>);
  if (variant == 0 && (e = ensure_dyn_smem<landmark8_kernel<DH, false, false>>(smem, dev)) == cudaSuccess) launch(landmark8_kernel<DH, false, false>);
  if (e != cudaSuccess) return e;
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_landmarks(const __nv_bfloat16* keys, __nv_bfloat16* landmarks, float* min_cos, int G, int batch, int T,
                             int H_kv, int d_h, int c, float rope_base, cudaStream_t s) {
  const int n_c = (T + c - 1) / c;
  const int tpr = H_kv * d_h / 16;                        // threads per key row
  if (tpr > kLmThreads || kLmThreads % tpr != 0) return cudaErrorInvalidValue;
  if (c == 8) {                                           // the default chunk has a kernel of its own
    const cudaError_t e = d_h == 128 ? launch_landmark8<128>(keys, landmarks, min_cos, G, batch, T, H_kv, rope_base, s)
                                     : launch_landmark8<64>(keys, landmarks, min_cos, G, batch, T, H_kv, rope_base, s);
    count_launch(kFamLandmarks);
    return e;
  }
  const int cpc = c >= kLmRows ? 1 : kLmRows / c;
  const dim3 grid((n_c + cpc - 1) / cpc, G, batch);
  const int use_rope = rope_base > 0.0f ? 1 : 0;
  if (d_h == 128)
    landmark_kernel<128><<<grid, kLmThreads, 0, s>>>(keys, landmarks, min_cos, G, batch, T, H_kv, c, n_c, cpc,
                                                     (double)rope_base, use_rope);
  else
    landmark_kernel<64><<<grid, kLmThreads, 0, s>>>(keys, landmarks, min_cos, G, batch, T, H_kv, c, n_c, cpc,
                                                    (double)rope_base, use_rope);
  count_launch(kFamLandmarks);
  return cudaGetLastError();
}

}  // namespace xkv
