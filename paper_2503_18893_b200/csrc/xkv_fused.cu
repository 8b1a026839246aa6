// Selective reconstruction (Sec. 3.2, Eq. 3) fused with decode attention over the rebuilt rows: the
// tensor-core path.  One persistent CTA per SM walks a contiguous range of 128-row tiles of the selected
// sets; a problem is one (layer, sequence, KV head).
//
// Per tile (128 selected rows S_t of one problem, j indexes the tile's rows, m the rank dimension):
//   keys    K_hat[j][d] = sum_m A_k[S_t[j]][m] B_k[m][d]       tcgen05.mma, M = rows, N = d_h, fp32 in TMEM
//           z[h][j]     = scale * <q_h, rope(K_hat[j])>          four lanes of a warp share a rebuilt key row
//           p[h][j]     = exp(z - running max)                   online softmax; p is handed on as bf16
//   values  W[m][h]    += sum_j A_v[S_t[j]][m] p[h][j]           tcgen05.mma, M = 128 rank columns, N = heads
// and once per problem, after the segments have been merged,  out_h = (W[:, h] / l_h)^T B_v.
// This is Eq. 3 for the values with the product re-associated: sum_j p_j (A_v[S_j] B_v) = (sum_j p_j A_v[S_j]) B_v,
// so the rebuilt value rows are consumed in factored form and never materialised.  Rebuilt key rows live in
// TMEM only.  Every gathered byte is written to shared memory once and read by the tensor core once.
//
// Warp roles: 0-3 key epilogue, 4-7 value epilogue, then gather producers, half of them for the key stream and half for
// the value stream (cp.async of the selected rows of A_k / A_v into two rings of 16 KB slabs, one per stream), then one
// warp of MMA issue for the key phases, one TMA loader of the B_k slabs (a short ring: they come from L2) and one warp of
// MMA issue for the value phases.  The two streams are coupled only through the data: a value phase needs the weights that the key
// epilogue derives from the same tile's key phase.  Slots are released in pairs by tcgen05.commit; every barrier
// has one producer side and waiters that see each of its phases in order, so that one parity bit per waiter is
// enough.  Every wait is bounded; a wait that runs out raises XKV_FLAG_TIMEOUT and the CTA winds down.
// The kernel starts under programmatic dependent launch: set-up overlaps the tail of the selection kernels.
//
// Diagnostic counters (cycles, per CTA, 64 words; see xkv_debug_read_profile): 0 key-stream producer total, 1-3 its
// waits (rotary/position buffers, positions, ring), 4 tiles; 48 value-stream producer total, 50-51 its waits
// (positions, ring); key-phase MMA warp: 8 total, 9 accumulator wait, 11 rows and B slabs, 12 issue;
// value-phase MMA warp: 40 total, 41 accumulator wait, 43 row ring, 44 issue, 45 weights; 17 loader wait;
// 24 key epilogue total, 25 positions, 26 accumulator, 27 group barrier, 28 weights buffer; 32 value epilogue
// total, 33 accumulator.
#include <cuda.h>

#include "xkv_gather.h"
#include "xkv_internal.cuh"
#include "xkv_ptx.cuh"

namespace xkv {

namespace {

using namespace ptx;

constexpr int kTile = 128;                       // selected rows per tile
constexpr int kSlabBytes = kTile * 128;          // 128 rows x 64 bf16 (one 128-byte swizzle row each)
// Gather producers: four warps (two per stream) issue asynchronous copies; eight where the rows are dequantised on the way,
// which is instruction work of the producers (4-bit bases at T = 131072, k = 4096: step 111.8 us with four, 93.7 with eight).
constexpr int prod_warps(int quant) { return quant ? 8 : 4; }
constexpr int fused_threads(int quant) { return (11 + prod_warps(quant)) * 32; }
constexpr int kSmemLimit = 227 * 1024;
constexpr int kPBytes = 2 * 16 * 128;            // softmax weights of a tile as a bf16 MMA operand: [2][16 heads][64 rows]
constexpr int kMaxBlocks = 8;                    // 128-column blocks of r_v that fit the TMEM accumulators
constexpr unsigned long long kWaitLimitNs = 250000000ull;    // a wait that lasts a quarter of a second has failed
constexpr float kLog2e = 1.4426950408889634f;
constexpr float kLn2 = 0.6931471805599453f;

struct Sched {
  int l0;            // first layer of the call
  int tpp;           // tiles per problem = ceil(k_cap / 128)
  int n_tiles;       // problems * tpp
  int n_ctas;
  int share, extra;  // tiles of a CTA; the first `extra` CTAs take one more
  int n_slots;       // partial slots per problem
  int k_cap;
  unsigned long long* prof;   // diagnostic counters [n_ctas][64] or nullptr
};

struct Walk {        // a CTA's tiles: [begin, end), the first problem's part ends at next
  int begin, end, next;
  int py, ti, l, b, g;   // the first problem: ordinal, tile in it, layer, sequence, head
  int seg;           // this CTA's segment of it
  unsigned loaded;   // pairs of B_k slabs that the loader has requested, for the wind-down
};
struct Bars {        // offsets (in 8-byte words) into the barrier array
  int full, fullv, emptyk, emptyv, kfull, kempty, wfull, wempty, pfull, rfree, posfull, vfree, grp, drain, total;
};
__host__ __device__ constexpr Bars bar_layout(int pk, int pv) {   // slot pairs of the key ring, of the value ring
  Bars b{};
  // one barrier per slot pair and direction: the issuing warp waits once per pair, for everything the pair holds
  b.full = 0; b.emptyk = pk; b.fullv = 2 * pk; b.emptyv = b.fullv + pv; b.kfull = b.emptyv + pv;
  b.kempty = b.kfull + 2; b.wfull = b.kempty + 2; b.wempty = b.wfull + 2; b.pfull = b.wempty + 2;
  b.rfree = b.pfull + 2; b.posfull = b.rfree + 2; b.vfree = b.posfull + 4; b.grp = b.vfree + 4; b.drain = b.grp + 1; b.total = b.drain + 2;
  return b;
}

// CTA i owns tiles [first_tile(i), first_tile(i + 1)); cta_of_tile is the owner of tile t.  32-bit divisions by numbers of
// the host: three 64-bit ones behind the dependency wait held a CTA's first gather up.
__device__ __forceinline__ int first_tile(const Sched& sc, int i) { return i * sc.share + min(i, sc.extra); }
__device__ __forceinline__ int cta_of_tile(const Sched& sc, int t) {
  const int split = sc.extra * (sc.share + 1);
  return t < split ? t / (sc.share + 1) : sc.extra + (t - split) / sc.share;
}

// PROF = false: `prof` is a compile-time null pointer and every diagnostic branch of the kernel folds away (the
// loops of the kernel have to stay small: the warps of a scheduler share its instruction cache).
template <bool PROF>
struct CtxT {
  volatile int* abort;
  unsigned int* flags;
  unsigned long long* prof;   // per-CTA diagnostic counters (cycles)
};
template <>
struct CtxT<false> {
  volatile int* abort;
  unsigned int* flags;
  static constexpr unsigned long long* prof = nullptr;
};
__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
// Bounded wait on an mbarrier phase.  Returns false if another thread of the CTA has given up, or if the
// phase does not complete within kWaitLimitNs (then this thread raises the flag and makes the others give up).
// The polling loop is one out-of-line function: the kernel's loops wait in dozens of places and have to stay
// small (the warps of a scheduler share its instruction cache).
__device__ __noinline__ bool wait_bar_slow(volatile int* abort_flag, unsigned int* flags, uint32_t bar, uint32_t parity) {
  const unsigned long long t0 = global_ns();
  // abort_flag[1] holds the limit in units of 2^16 ns (0: the default)
  const unsigned long long limit = abort_flag[1] ? ((unsigned long long)abort_flag[1] << 16) : kWaitLimitNs;
  for (uint32_t i = 1;; ++i) {
    if (mbar_try_wait(bar, parity)) return true;
    if ((i & 63u) == 0u) {
      if (*abort_flag) return false;
      if (global_ns() - t0 > limit) break;
    }
  }
  *abort_flag = 1;
  atomicOr(flags, XKV_FLAG_TIMEOUT);
  return false;
}
template <class Ctx>
__device__ __forceinline__ bool wait_bar_raw(const Ctx& c, uint32_t bar, uint32_t parity) {
  if (mbar_try_wait(bar, parity)) return true;
  return wait_bar_slow(c.abort, c.flags, bar, parity);
}
// `slot` >= 0 (passed warp-uniformly by one warp per role when diagnostics are on) adds the cycles waited.
template <class Ctx>
__device__ __forceinline__ bool wait_bar(const Ctx& c, uint32_t bar, uint32_t parity, int slot = -1) {
  if (c.prof == nullptr || slot < 0) return wait_bar_raw(c, bar, parity);
  const long long c0 = clock64();
  const bool r = wait_bar_raw(c, bar, parity);
  if ((threadIdx.x & 31) == 0) atomicAdd(c.prof + slot, (unsigned long long)(clock64() - c0));
  return r;
}

// The queries in shared memory, fp32: [head][d_h / 4] units of 16 bytes, unit u = dimensions {2u, 2u + 1, d_h/2 + 2u,
// d_h/2 + 2u + 1}, which is what two rotary pairs (i, i + d_h/2) are multiplied with.

__device__ __forceinline__ void mma_tf32(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// Logits of the 32 rebuilt key rows of a warp against NR query heads: rotate the (i, i + HALF) pairs, multiply.
// Four lanes share a row: lane 4g + t reads rows g, g + 8, g + 16, g + 24 and of every eight dimensions 2t and 2t + 1 (the
// 16x256b form of tcgen05.ld), so that a query or table entry it loads serves four rows, and two dimensions side by side are
// the operands of one packed instruction.  One warp per scheduler issues a multiply-add every two cycles at best, so what
// bounds this is their number: 8 a pair for the angles and the rotation, and 2 for every head.
// MMA: the heads (rounded up to eights) are multiplied by mma.sync instead: the rotated values are where an operand of
// m16n8k8 wants them.  The queries are bf16 and thus exact as tf32; a key element goes in as two parts, its nearest value of 11
// bits and the rest, 12 bits and a sign, of which the tensor core keeps 11: at most 2^-23 of the element is lost.  The tensor
// core cuts its sums off instead of rounding them, so a sum runs over sixteen dimensions only and is added on in fp32: one sum
// over all of them (32 steps), and an upper part that was cut off too, had logits of single rows off by 1.2 to 1.5 (rms,
// in 2^-24 of sum |q k|; d_h 64 and 128); now 0.24 to 0.33, a multiply-add per element and head in fp32 0.36 to 0.51, the
// packed form 0.24.  Seven heads 123.9 -> 122.5 us a step with it, 4-bit bases 87.2 -> 87.2, 32768 rows by layer 112.1 -> 112.3; a call
// with sixteen heads 72.1 -> 75.5 and with 3-bit bases and four heads 50.0 -> 52.2: every pass waits for its four products.  (The
// sums added a pass later, so that nothing waits: 3-bit 52.6, seven heads 124.0; the rounding by cvt.rna.tf32: 123.9.)
// Which one: without MMA only four heads and bf16 bases have registers for the sums (eight heads 157.4 us a step of eight
// sequences of 65536 rows where a row per lane takes 151.9, 4-bit bases 92.5 where it takes 88.3; with MMA, seven heads 129.4 ->
// 122.5 and 4-bit bases 88.2 -> 87.1), and there it is the better one from two tiles per CTA on, where shared memory and the tensor
// pipe are all but busy: 131072 rows 78.3 -> 75.4 us a step from a row per lane, with MMA 78.6 -> 79.2; four sequences of them 268.3
// -> 252.4, with MMA 270.4 -> 268.7; rank 1024 and a budget of 16384 316.5 -> 311.9.  A call of 37 problems
// and 1, 2, 3, 7 tiles per CTA, MMA / without: four heads of 128, rank 512 17.4 / 17.4, 22.0 / 21.0, 26.3 / 24.2, 44.2 /
// 38.8 us; rank 64 13.2 / 13.2, 16.0 / 16.0, 18.5 / 18.6, 29.1 / 29.3; rank 1024 23.5 / 23.6, 33.4 / 33.0, 41.6 / 41.3, 67.5 /
// 66.9; one head, rank 512 15.8 / 16.1, 20.4 / 19.4, 24.6 / 22.7, 42.1 / 36.7; four heads of 64, rank 256 14.4 / 14.3, 16.9 / 16.4,
// 19.6 / 18.4, 29.8 / 26.5.
// hi: the coarse rotary entries of the warp's four 8-row chunks, 16-byte units; lo: the fine ones of position g of a
// chunk, units swizzled by `swz`; q_s: the queries.  On return a lane holds the logits of row g + 8t.
template <int DH, int NR, bool MMA>
__device__ __forceinline__ void quad_logits(uint32_t acc, const ulonglong2* __restrict__ hi, const ulonglong2* __restrict__ lo,
                                            int swz, const uint4* __restrict__ q_s, int lane, float (&z)[NR]) {
  constexpr int HALF = DH / 2, UN = HALF / 2;            // units of a rotary row, of a head
  constexpr int NT = (NR + 7) / 8;                       // groups of eight heads
  constexpr unsigned long long kNeg2 = 0x8000000080000000ull;
  const int t = lane & 3, g = lane >> 2;
  float c[NT][2][4];                                     // MMA: [.][rows g, g + 8 | g + 16, g + 24][heads 2t, 2t + 1 of either]
  u64 s[MMA ? 1 : 4][NR];                                // else: [row][head], sums of the even and of the odd dimensions
#pragma unroll
  for (int n = 0; n < NT; ++n)
#pragma unroll
    for (int i = 0; i < 8; ++i) c[n][i >> 2][i & 3] = 0.0f;
#pragma unroll
  for (int r = 0; r < (MMA ? 1 : 4); ++r)
#pragma unroll
    for (int h = 0; h < NR; ++h) s[r][h] = 0ull;
#pragma unroll 1
  for (int jj = 0; jj < HALF / 8; ++jj) {
    uint32_t xa[2][4], xb[2][4];                         // [16 rows][row g: 2 dimensions, row g + 8: 2]
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const uint32_t at = acc + ((uint32_t)i << 20) + (uint32_t)(jj * 8);
      tmem_ld_quad(at, xa[i]);
      tmem_ld_quad(at + (uint32_t)HALF, xb[i]);
    }
    const int u = jj * 4 + t;
    const ulonglong2 f = lo[u ^ swz];                    // {cosines, sines} of two pairs
    ulonglong2 a[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) a[r] = hi[r * UN + u];
    uint4 qv[NT];                                        // head 8 n + g (heads beyond NR: whatever, their columns are not read)
#pragma unroll
    for (int n = 0; n < NT && MMA; ++n) qv[n] = q_s[(8 * n + (NR < 8 ? g & (NR - 1) : g)) * UN + u];
#pragma unroll
    for (int i = 0; i < 2; ++i) tc_wait_ld_nb(xa[i], xb[i]);
    const u64 fn = f.y ^ kNeg2;
    u64 r1[4], r2[4];                                    // the rotated pairs, either half
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const u64 cs = fma2(a[r].y, fn, mul2(a[r].x, f.x));            // cos(x + y)
      const u64 sn = fma2(a[r].x, f.y, mul2(a[r].y, f.x));           // sin(x + y)
      const u64 x1 = pack2u(xa[r >> 1][2 * (r & 1)], xa[r >> 1][2 * (r & 1) + 1]);
      const u64 x2 = pack2u(xb[r >> 1][2 * (r & 1)], xb[r >> 1][2 * (r & 1) + 1]);
      r1[r] = fma2(x2, sn ^ kNeg2, mul2(x1, cs));
      r2[r] = fma2(x1, sn, mul2(x2, cs));
    }
    if constexpr (!MMA) {
#pragma unroll
      for (int h = 0; h < NR; ++h) {
        const ulonglong2 qh = reinterpret_cast<const ulonglong2*>(q_s)[h * UN + u];
#pragma unroll
        for (int r = 0; r < 4; ++r) s[r][h] = fma2(qh.x, r1[r], s[r][h]);
#pragma unroll
        for (int r = 0; r < 4; ++r) s[r][h] = fma2(qh.y, r2[r], s[r][h]);
      }
      continue;
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      uint32_t h1[4], h2[4], l1[4], l2[4];               // [row g: 2 dimensions, row g + 8: 2], either half; upper and lower parts
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const float2 p1 = unpack2(r1[2 * i + k]), p2 = unpack2(r2[2 * i + k]);
        const float v[4] = {p1.x, p1.y, p2.x, p2.y};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const uint32_t up = (__float_as_uint(v[e]) + 0x1000u) & 0xffffe000u, rest = __float_as_uint(v[e] - __uint_as_float(up));
          if (e < 2) { h1[2 * k + e] = up; l1[2 * k + e] = rest; } else { h2[2 * k + e - 2] = up; l2[2 * k + e - 2] = rest; }
        }
      }
#pragma unroll
      for (int n = 0; n < NT; ++n) {
        // sums of sixteen dimensions, lower parts first, added in fp32
        float d[4] = {0.0f, 0.0f, 0.0f, 0.0f};
        mma_tf32(d, l1[0], l1[2], l1[1], l1[3], qv[n].x, qv[n].y);
        mma_tf32(d, l2[0], l2[2], l2[1], l2[3], qv[n].z, qv[n].w);
        mma_tf32(d, h1[0], h1[2], h1[1], h1[3], qv[n].x, qv[n].y);
        mma_tf32(d, h2[0], h2[2], h2[1], h2[3], qv[n].z, qv[n].w);
#pragma unroll
        for (int e = 0; e < 4; ++e) c[n][i][e] += d[e];
      }
    }
  }
  const bool up1 = (t & 1) != 0, up2 = (t & 2) != 0;
  if constexpr (!MMA) {
    // sums over the four lanes of a row, folded by halving: a lane ends with one row
#pragma unroll
    for (int h = 0; h < NR; ++h) {
      float v[4], w[2];
#pragma unroll
      for (int r = 0; r < 4; ++r) { const float2 p = unpack2(s[r][h]); v[r] = p.x + p.y; }
#pragma unroll
      for (int r = 0; r < 2; ++r) w[r] = (up2 ? v[r + 2] : v[r]) + __shfl_xor_sync(0xffffffffu, up2 ? v[r] : v[r + 2], 2);
      z[h] = (up1 ? w[1] : w[0]) + __shfl_xor_sync(0xffffffffu, up1 ? w[0] : w[1], 1);
    }
    return;
  }
  // transpose among the four lanes of a row: from heads 2t, 2t + 1 of four rows to all heads of row g + 8t
#pragma unroll
  for (int n = 0; n < NT; ++n) {
    float w[2][2][2];                                    // [heads 2 (t & 1), + 1 | those and 4][row][head of the pair]
#pragma unroll
    for (int k = 0; k < 2; ++k)
#pragma unroll
      for (int x = 0; x < 2; ++x) {
        const float low = c[n][0][2 * k + x], high = c[n][1][2 * k + x];         // rows k, k + 2
        const float mine = up2 ? high : low, got = __shfl_xor_sync(0xffffffffu, up2 ? low : high, 2);
        w[0][k][x] = up2 ? got : mine;
        w[1][k][x] = up2 ? mine : got;
      }
#pragma unroll
    for (int p = 0; p < 2; ++p)
#pragma unroll
      for (int x = 0; x < 2; ++x) {
        if (8 * n + 4 * p >= NR) continue;
        const float mine = up1 ? w[p][1][x] : w[p][0][x], got = __shfl_xor_sync(0xffffffffu, up1 ? w[p][0][x] : w[p][1][x], 1);
        z[8 * n + 4 * p + x] = up1 ? got : mine;
        z[8 * n + 4 * p + 2 + x] = up1 ? mine : got;
      }
  }
}

// Rotary rows are multiples of 128 bytes.  Unit u of a fine row is kept at u ^ lo_swz(row): the eight lanes of a quarter warp
// hit all banks once, be they two neighbouring rows of four units (quad_logits) or the same unit of eight rows (key_logits_rows).
__host__ __device__ constexpr int lo_swz(int row) { return ((row & 1) << 2) | (row >> 1); }

// The same for the variants that ordinary tiles do not take, a row per lane, out of line, because the key epilogue's loop has to
// stay small (the four warps of a scheduler run four different loops and share its instruction cache: 32 pairs unrolled in it
// took 77 us a call, 8 pairs 73, 4 pairs 71).  Rotary rows: none; the staged ones (hi, lo: shared-memory addresses, units of lo
// swizzled by swz), where 8-row groups share a coarse row, in whatever order; the handle's (hi, lo: addresses) where they share
// none, or the fine table is not staged.  (Rows of whole chunks in any order, from the handle's tables -> from the staged ones: four
// heads, 131072 rows, budget 4096 69.4 -> 40.8 us, in order 40.0; seven heads, eight sequences of 65536 rows 135.8 -> 73.0, in
// order 67.5; sixteen heads 109.3 -> 82.4, in order 74.4; 4-bit bases, four heads 73.1 -> 53.2, in order 50.8.)
// On return a lane holds the logits of the row of its own TMEM lane.
enum RowTables { kNoTables, kHandleTables, kStagedTables };
template <int NR>
struct LogitsOut { float z[NR]; };
__device__ __forceinline__ ulonglong2 lds_u64x2(uint32_t addr) {
  ulonglong2 v;
  asm volatile("ld.shared.v2.u64 {%0, %1}, [%2];" : "=l"(v.x), "=l"(v.y) : "r"(addr));
  return v;
}
template <int DH, int NR, int QUANT, int TABLES>
__device__ __noinline__ LogitsOut<NR> key_logits_rows(uint32_t acc, unsigned long long hi, unsigned long long lo, int swz,
                                                      const ulonglong2* __restrict__ q_s) {
  constexpr int HALF = DH / 2;
  constexpr unsigned long long kNeg2 = 0x8000000080000000ull;
  // Two dimensions per instruction where the sums have registers: not with sixteen heads, and with eight over codes (96 registers
  // a thread) only without tables.  One by one -> packed: 4-bit bases, seven heads, no RoPE 83.0 -> 80.3 us; rows of no chunk,
  // four heads 70.7 -> 69.9, over codes 78.0 -> 75.7; seven heads 133.3 -> 132.4, but over codes 145 -> 157.
  constexpr bool PACKED = NR <= 8 && !(NR == 8 && QUANT != 0 && TABLES != kNoTables);
  LogitsOut<NR> o;
  u64 s[PACKED ? NR : 1];
#pragma unroll
  for (int h = 0; h < NR; ++h) o.z[h] = 0.0f;
#pragma unroll
  for (int h = 0; h < (PACKED ? NR : 1); ++h) s[h] = 0ull;
#pragma unroll 1
  for (int u = 0; u < HALF / 2; u += 2) {                // four rotary pairs per pass
    uint32_t xa[4], xb[4];
    tmem_ld4_nb(acc + (uint32_t)(2 * u), xa);
    tmem_ld4_nb(acc + (uint32_t)(HALF + 2 * u), xb);
    ulonglong2 a[2], f[2];
    if (TABLES == kHandleTables) {
#pragma unroll
      for (int v = 0; v < 2; ++v) {
        a[v] = __ldg(reinterpret_cast<const ulonglong2*>(hi) + u + v);
        f[v] = __ldg(reinterpret_cast<const ulonglong2*>(lo) + u + v);
      }
    }
    if (TABLES == kStagedTables) {
#pragma unroll
      for (int v = 0; v < 2; ++v) {
        a[v] = lds_u64x2((uint32_t)hi + (uint32_t)(u + v) * 16u);
        f[v] = lds_u64x2((uint32_t)lo + (uint32_t)((u + v) ^ swz) * 16u);
      }
    }
    tc_wait_ld_nb(xa, xb);
#pragma unroll
    for (int v = 0; v < 2; ++v) {
      u64 r1 = pack2u(xa[2 * v], xa[2 * v + 1]), r2 = pack2u(xb[2 * v], xb[2 * v + 1]);
      if (TABLES != kNoTables) {
        const u64 cs = fma2(a[v].y, f[v].y ^ kNeg2, mul2(a[v].x, f[v].x));       // cos(x + y)
        const u64 sn = fma2(a[v].x, f[v].y, mul2(a[v].y, f[v].x));               // sin(x + y)
        const u64 x1 = r1, x2 = r2;
        r1 = fma2(x2, sn ^ kNeg2, mul2(x1, cs));
        r2 = fma2(x1, sn, mul2(x2, cs));
      }
      // heads in groups of four: their multiply-adds are independent (one head after the other is a chain)
#pragma unroll
      for (int h0 = 0; h0 < NR; h0 += 4) {
        ulonglong2 qv[4];
#pragma unroll
        for (int h = 0; h < 4; ++h) qv[h] = q_s[(h0 + h) * (DH / 4) + u + v];
        if constexpr (PACKED) {
#pragma unroll
          for (int h = 0; h < 4; ++h) s[h0 + h] = fma2(qv[h].x, r1, s[h0 + h]);
#pragma unroll
          for (int h = 0; h < 4; ++h) s[h0 + h] = fma2(qv[h].y, r2, s[h0 + h]);
        } else {
          const float2 p1 = unpack2(r1), p2 = unpack2(r2);
#pragma unroll
          for (int h = 0; h < 4; ++h) o.z[h0 + h] = fmaf(unpack2(qv[h].x).x, p1.x, o.z[h0 + h]);
#pragma unroll
          for (int h = 0; h < 4; ++h) o.z[h0 + h] = fmaf(unpack2(qv[h].y).x, p2.x, o.z[h0 + h]);
#pragma unroll
          for (int h = 0; h < 4; ++h) o.z[h0 + h] = fmaf(unpack2(qv[h].x).y, p1.y, o.z[h0 + h]);
#pragma unroll
          for (int h = 0; h < 4; ++h) o.z[h0 + h] = fmaf(unpack2(qv[h].y).y, p2.y, o.z[h0 + h]);
        }
      }
    }
  }
  if constexpr (PACKED) {
#pragma unroll
    for (int h = 0; h < NR; ++h) { const float2 p = unpack2(s[h]); o.z[h] = p.x + p.y; }
  }
  return o;
}

// Slots of the ring of gathered key rows, of the ring of the B_k slabs that go with them (slab pair by slab pair).
constexpr int kKeySlots = 4;
constexpr int kBarWords = 48;
constexpr int kWalkInts = 12;
static_assert(sizeof(Walk) <= kWalkInts * sizeof(int), "walk");
// Shared memory besides the rings: weights, rotary rows, queries, positions, barriers.
template <int DH, int NR>
__host__ __device__ constexpr int misc_smem_bytes() {
  return (int)(2 * kPBytes + sizeof(float2) * (2 * 16 + 8) * (DH / 2) + sizeof(float) * (NR * DH + 2 * NR + 8 * NR) +
               sizeof(int) * (4 * kTile + 8 + kWalkInts) + 8 * kBarWords + 16);
}
// Slots of the ring of gathered value rows: whatever fits beside those two, at most as many.
template <int DH, int NR>
__host__ __device__ constexpr int value_slots() {
  const int fit = ((kSmemLimit - 1024 - misc_smem_bytes<DH, NR>() - 2 * kKeySlots * kSlabBytes) / kSlabBytes) & ~1;   // even: released in pairs
  return fit < kKeySlots ? fit : kKeySlots;
}

// NR: query heads per KV head rounded up to 4, 8 or 16.  WB: most 128-column blocks of r_v (registers of the
// value epilogue): NR * WB <= 64.
// MMA: how the key epilogue multiplies (quad_logits).
// QUANT = 4 or 3: the token bases are gathered from 4-bit or 3-bit codes (xkv_group_set_quantized_bases) and
// dequantised by the producer warps on their way into the rings; 0: bf16 bases.
template <int DH, int NR, int WB, bool PROF, int QUANT, bool MMA>
__global__ void __launch_bounds__(fused_threads(QUANT), 1)
sr_fused_kernel(const __grid_constant__ CUtensorMap bk_map, GroupDev dev, Sched sc, const __nv_bfloat16* __restrict__ q,
                const int32_t* __restrict__ sel_idx, const int32_t* __restrict__ sel_cnt) {
  extern __shared__ uint8_t smem_raw[];
  constexpr int HALF = DH / 2;
  constexpr int kThreads = fused_threads(QUANT), PW = prod_warps(QUANT), SPT = PW * 16;   // SPT: producer threads per stream
  constexpr int kWarpK = 8 + PW, kWarpB = kWarpK + 1, kWarpV = kWarpK + 2;                // key MMA, B loader, value MMA
  // (through a shuffle, so that the compiler knows it to be the same in all lanes)
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* gen = smem_raw + (base - smem_u32(smem_raw));
  // rings of slabs: SK of gathered key rows, SV of gathered value rows, SK of B_k slabs (all even, all may be in flight)
  constexpr int SK = kKeySlots, SV = value_slots<DH, NR>(), S = SK + SV;
  static_assert(SK >= 2 && SV >= 2 && SK % 2 == 0 && SV % 2 == 0, "rings");
  const uint32_t bring = base + (uint32_t)S * kSlabBytes;                         // B-slab ring
  // carve-up after the rings
  uint8_t* P_gen = gen + (size_t)(S + SK) * kSlabBytes;                          // [2][kPBytes] bf16 weights (MMA operand)
  const uint32_t P_addr = base + (uint32_t)(S + SK) * kSlabBytes;
  constexpr int UN = HALF / 2;                                                   // 16-byte units {cos, cos, sin, sin} of a rotary row
  float4* hi_s = reinterpret_cast<float4*>(P_gen + 2 * kPBytes);                 // [2][16][UN] coarse rotary rows
  float4* lo_s = hi_s + 2 * 16 * UN;                                             // [8][UN]     fine rotary rows, unit u of row i at u ^ lo_swz(i)
  float* q_s = reinterpret_cast<float*>(lo_s + 8 * UN);                          // [NR][DH], see quad_logits
  float* alpha_s = q_s + NR * DH;                                                // [2][NR]
  float* red_s = alpha_s + 2 * NR;                                               // [2][4][NR]
  int* pos_s = reinterpret_cast<int*>(red_s + 2 * 4 * NR);                       // [4][128]
  int* algn_s = pos_s + 4 * kTile;                                               // [2][4]
  Walk* walk_s = reinterpret_cast<Walk*>(algn_s + 8);
  uint64_t* bars = reinterpret_cast<uint64_t*>(algn_s + 8 + kWalkInts);
  constexpr Bars bl = bar_layout(SK / 2, SV / 2);
  static_assert(bl.total <= kBarWords, "barrier space");
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + bl.total);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  const uint32_t bar0 = smem_u32(bars);
  auto BAR = [&](int word) { return bar0 + 8u * (uint32_t)word; };
  CtxT<PROF> ctx;
  ctx.abort = abort_flag;
  ctx.flags = dev.flags;
  if constexpr (PROF) ctx.prof = sc.prof ? sc.prof + (size_t)blockIdx.x * 64 : nullptr;
  // the staged rotary path needs the fine table to cover exactly 8 positions
  const bool rope_smem = dev.use_rope && dev.rope_shift == 3;
  // both phases are padded to an even number of 64-column slabs so that slabs pair up inside ring-slot pairs
  const int nks_k = (dev.r_k + 63) >> 6, nks_v = (dev.r_v + 63) >> 6;
  const int nst_k = (nks_k + 1) & ~1, nst_v = (nks_v + 1) & ~1;

  const int per_layer = dev.batch * dev.H_kv;
  const int n_rep = dev.n_rep;
  if (tid == 64) {     // the CTA's range, once (divisions), to shared memory: only the walk's rare steps look at it again
    const int first = first_tile(sc, blockIdx.x), py = first / sc.tpp, ti = first - py * sc.tpp;
    walk_s->begin = first; walk_s->end = first_tile(sc, blockIdx.x + 1);
    walk_s->next = min(walk_s->end, first - ti + sc.tpp);
    walk_s->py = py; walk_s->ti = ti;
    walk_s->g = py % dev.H_kv; walk_s->b = (py / dev.H_kv) % dev.batch; walk_s->l = sc.l0 + py / per_layer;
    walk_s->seg = (int)blockIdx.x - cta_of_tile(sc, py * sc.tpp);
  }

  if (tid == 0) {
    for (int s = 0; s < SK / 2; ++s) { mbar_init(BAR(bl.full + s), SPT + 1); mbar_init(BAR(bl.emptyk + s), 1); }
    for (int s = 0; s < SV / 2; ++s) { mbar_init(BAR(bl.fullv + s), SPT); mbar_init(BAR(bl.emptyv + s), 1); }
    for (int b = 0; b < 2; ++b) {
      mbar_init(BAR(bl.kfull + b), 1); mbar_init(BAR(bl.kempty + b), 128);
      mbar_init(BAR(bl.wfull + b), 1); mbar_init(BAR(bl.wempty + b), 128);
      mbar_init(BAR(bl.pfull + b), 128);
      mbar_init(BAR(bl.rfree + b), 128);
    }
    for (int b = 0; b < 4; ++b) { mbar_init(BAR(bl.posfull + b), SPT); mbar_init(BAR(bl.vfree + b), SPT); }
    mbar_init(BAR(bl.grp), 128);
    mbar_init(BAR(bl.drain), 1); mbar_init(BAR(bl.drain + 1), 1);
    abort_flag[0] = 0;
    // an injected fault: give up after about a millisecond
    abort_flag[1] = (dev.inject & (XKV_INJECT_FUSED_NO_B | XKV_INJECT_FUSED_NO_ROWS)) ? 16 : 0;
    fence_mbar_init();
  }
  if (rope_smem) {
    for (int i = tid; i < 8 * UN; i += kThreads) lo_s[(i / UN) * UN + ((i % UN) ^ lo_swz(i / UN))] = dev.rope_lo[i];
  }
  // weights of heads that do not exist stay zero for the whole kernel
  for (int i = tid; i < 2 * kPBytes / 4; i += kThreads) reinterpret_cast<uint32_t*>(P_gen)[i] = 0u;
  fence_proxy_async();
  if (warp == kWarpK) {
    tmem_alloc(smem_u32(tmem_slot), 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  // everything above is independent of the inputs; the selection (or whatever wrote q and the index sets) comes
  // from earlier kernels of the stream
  grid_dependency_wait();
  grid_dependency_launch();

  // Walks this CTA's tiles, skipping tiles that start at or beyond the problem's row count.
  // The tiles of the range's first problem, which are the end of it wherever the range goes on to another problem, come
  // last: the rows of a selection are ascending, so the CTAs then move through the contexts together (each from the start
  // of a problem, or close to it), and a row that several heads of a sequence selected is asked for by all of them while it
  // is in L2.  Four sequences of 131072 rows, budget 4096: 802 -> 400 MB from DRAM (340 MB are distinct), 141 -> 124 us;
  // 65536 rows, budget 16384, rank 1024: 340 -> 321 us a step.
  struct TileIter {
    int t, stop, py, ti, cnt, l, b, g, pyn; long long prob;   // t: tile ordinal of the call; pyn/ti: problem and tile in it
  };
  auto iter_begin = [&](TileIter& it_) {
    const bool more = walk_s->next < walk_s->end;
    it_.t = (more ? walk_s->next : walk_s->begin) - 1; it_.stop = walk_s->end;
    it_.py = -1; it_.cnt = 0; it_.prob = 0; it_.pyn = walk_s->py; it_.ti = (more ? sc.tpp : walk_s->ti) - 1;
    it_.l = walk_s->l; it_.b = walk_s->b; it_.g = walk_s->g;
  };
  // advance to the next non-empty tile; returns false at the end of the range.  Whenever the walk moves to a new
  // problem (also one whose tiles are all empty), `on_leave()` runs with the old problem still in `it_` (not before
  // the first one) and `on_enter()` with the new one, before its tiles.
  auto iter_next = [&](TileIter& it_, auto&& on_leave, auto&& on_enter) -> bool {
    for (;;) {
      if (++it_.t >= it_.stop) {
        if (it_.pyn == walk_s->py) return false;          // (the first problem's part is the last)
        it_.t = walk_s->begin; it_.stop = walk_s->next; it_.pyn = walk_s->py; it_.ti = walk_s->ti;
      } else if (++it_.ti == sc.tpp) {
        it_.ti = 0; ++it_.pyn;
      }
      const int py = it_.pyn;
      if (py != it_.py) {
        if (it_.py >= 0) on_leave();
        if (py == walk_s->py) {
          it_.l = walk_s->l; it_.b = walk_s->b; it_.g = walk_s->g;
        } else if (++it_.g == dev.H_kv) {
          it_.g = 0; if (++it_.b == dev.batch) { it_.b = 0; ++it_.l; }
        }
        it_.py = py;
        it_.prob = ((long long)it_.l * dev.batch + it_.b) * dev.H_kv + it_.g;
        it_.cnt = min(sel_cnt[it_.prob], sc.k_cap);
        on_enter();
      }
      if (it_.ti * kTile < it_.cnt) return true;
    }
  };
  auto no_op = []() {};
  // partial slot of the segment (this CTA's share) of problem ordinal py
  auto part_of = [&](int py, long long prob) {
    const int seg = py == walk_s->py ? walk_s->seg : 0;   // (later problems of the CTA start inside its range)
    return dev.part + ((size_t)prob * sc.n_slots + seg) * (size_t)n_rep * (dev.r_v + 2);
  };

  uint32_t pairs = 0;   // slot pairs that this thread (a producer, the loader) has begun to fill
  if (warp >= 8 && warp < kWarpK) {
    // =============================== producers: gather rows of A ===============================
    // Two independent streams with a ring of their own each: the first half of the producer warps (8-9, with quantised
    // bases 8-11) gather the rows of A_k of every tile into the key ring, the second half (10-11, 12-15) the same rows of
    // A_v into the value ring.  A stream waits only for releases of its own ring, so the key MMAs of consecutive tiles follow one another without waiting for the value phase that
    // sits between them in time (with one shared ring the key slabs of tile i+2 could not be requested before the
    // last value slab of tile i, which itself waited for the last key MMA of tile i+1).
    // Eight consecutive lanes copy the eight 16-byte pieces of one 128-byte row slab, so that every request of a
    // warp covers whole 128-byte lines; thread t of a stream serves rows (t>>3) + 8*i, i = 0..15.
    const bool kstream = warp < 8 + PW / 2;
    const int ts = (tid - 256) & (SPT - 1), pw = (warp - 8) & (PW / 2 - 1);
    const uint32_t c8 = (uint32_t)(ts & 7), r8 = (uint32_t)(ts >> 3);
    // rows r8 + 8*i share the swizzle phase r8; slab-relative destination of the i = 0 piece
    const uint32_t dst0 = r8 * 128u + ((c8 ^ r8) << 4);
    const int ps = (warp == 8) ? 0 : (warp == 8 + PW / 2 ? 48 : -1000);
    const long long role_t0 = clock64();
    int slot = 0;                     // position in this stream's ring
    uint32_t used = 0, rel_par = 0;   // per slot pair: filled before; parity of the release to wait for next
    int it = 0, pb = 0;               // tiles done; position buffer of the tile (four in rotation)
    bool ok = true;
    const int RS = kstream ? SK : SV;                           // slabs in this stream's ring
    const uint32_t ring0 = base + (kstream ? 0u : (uint32_t)SK * kSlabBytes) + dst0;
    const int bar_full = kstream ? bl.full : bl.fullv, bar_empty = kstream ? bl.emptyk : bl.emptyv;
    const int r = kstream ? dev.r_k : dev.r_v;
    const uint32_t row_bytes = (uint32_t)r * 2u;
    const int nst = kstream ? nst_k : nst_v;
    const __nv_bfloat16* Abase = kstream ? dev.A_k : dev.A_v;
    // one phase of one tile: the 64-column slabs of its gathered rows, two at a time (slots are released in
    // pairs, one tcgen05.commit per two slabs); ro: the tile rows of this thread
    auto issue_phase = [&](const uint32_t (&ro)[16], int b) {
      const char* Ab = reinterpret_cast<const char*>(Abase + (long long)b * dev.T * r) + c8 * 16u;
#pragma unroll 1
      for (int ks = 0; ks < nst; ks += 2) {
        const int pr = slot >> 1;
        const uint32_t bit = 1u << pr;
        if (used & bit) {             // wait for the release of the pair's previous occupant
          if (!wait_bar(ctx, BAR(bar_empty + pr), (rel_par >> pr) & 1u, ps + 3)) { ok = false; return; }
          rel_par ^= bit;
        }
        used |= bit;
        const uint32_t st = ring0 + (uint32_t)slot * kSlabBytes;
        // false in a ragged last slab or a padding slab: zero-fill (the source stays inside the row)
        const bool in0 = ks * 64 + (int)c8 * 8 < r, in1 = (ks + 1) * 64 + (int)c8 * 8 < r;
        const uint32_t n0 = in0 ? 16u : 0u, n1 = in1 ? 16u : 0u;
        const char* s0 = Ab + (in0 ? ks * 128 : 0);
        const char* s1 = Ab + (in1 ? ks * 128 + 128 : 0);
#pragma unroll
        for (int i = 0; i < 16; ++i) cp_async16(st + (uint32_t)i * 1024u, s0 + (size_t)ro[i] * row_bytes, n0);
#pragma unroll
        for (int i = 0; i < 16; ++i) cp_async16(st + kSlabBytes + (uint32_t)i * 1024u, s1 + (size_t)ro[i] * row_bytes, n1);
        cp_async_arrive_noinc(BAR(bar_full + pr));         // arrives when this thread's copies have landed
        ++pairs;
        slot += 2;
        if (slot == RS) slot = 0;
      }
    };
    // The same phase from 4-bit codes.  Four consecutive lanes share a tile row: lane q4 fetches the 16 bytes of
    // codes and the scale/offset word of one 32-column group of the slot pair (64 contiguous bytes per row and
    // request), turns them into 32 bf16 values (packed arithmetic, one rounding) and stores them as four 16-byte
    // units of the swizzled slab; a stream's 128 threads cover 32 rows per pass, 4 passes per pair.
    // What bounds it is instructions: every warp of a scheduler issues beside the key epilogue (of 13 k cycles a tile the key
    // stream waited 0.5 k for its ring).  Addresses are therefore worked out once, as one offset per row and one per
    // 16-byte unit, and a group's next codes are requested when it is converted, in the same registers.  131072 rows, budget
    // 4096, rank 512, 4 bits, kernel and merge: 70.7 us with the loads of a pair in front of its conversion, 66.6 behind that
    // of the pair before, 62.5 with the addresses.  Requesting the next tile's first codes from the last pair of a tile as
    // well, with its positions published a tile ahead, loses (68.6), and so do prefetches of its rows into L2 (74.7).
    const uint32_t q4 = (uint32_t)(ts & 3), rq = (uint32_t)(ts >> 2);
    constexpr int QP = 4;                                  // passes per slot pair
    // This lane's group lies in slab (q4 >> 1) of the pair, 16-byte units 4*(q4 & 1) .. +3 of the 128-byte row; here of
    // slot 0 and tile row rq.
    uint32_t unit[4];
    if constexpr (QUANT != 0) {
#pragma unroll
      for (int u = 0; u < 4; ++u)
        unit[u] = base + (kstream ? 0u : (uint32_t)SK * kSlabBytes) + (q4 >> 1) * kSlabBytes + rq * 128u + ((((q4 & 1u) * 4u + (uint32_t)u) ^ (rq & 7u)) << 4);
    }
    // gw: the first group of every row, counted over the sequence (the same for codes and parameters)
    auto issue_phase_q = [&](const uint32_t (&gw)[QP], int b) {
      const uint4* Cb = reinterpret_cast<const uint4*>((kstream ? dev.Aq_k : dev.Aq_v) + (size_t)b * dev.T * (size_t)(r >> 1));
      const uint32_t* Mb = (kstream ? dev.Am_k : dev.Am_v) + (size_t)b * dev.T * (size_t)(r >> 5);
      uint4 cw[QP];
      uint32_t mw[QP];
      auto fetch = [&](int ks, int i) {
        const uint32_t at = gw[i] + quant_group(ks, q4, r);
        // 4 bits: 16 bytes of codes and a separate scale/offset word; 3 bits: one 16-byte record {meta, w0, w1, w2}
        cw[i] = __ldg(Cb + at);
        if (QUANT == 4) mw[i] = __ldg(Mb + at);
      };
#pragma unroll
      for (int i = 0; i < QP; ++i) fetch(0, i);
#pragma unroll 1
      for (int ks = 0; ks < nst; ks += 2) {
        const int pr = slot >> 1;
        const uint32_t bit = 1u << pr;
        if (used & bit) {             // wait for the release of the pair's previous occupant
          if (!wait_bar(ctx, BAR(bar_empty + pr), (rel_par >> pr) & 1u, ps + 3)) { ok = false; return; }
          rel_par ^= bit;
        }
        used |= bit;
        uint32_t to[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) to[u] = unit[u] + (uint32_t)slot * kSlabBytes;
#pragma unroll
        for (int i = 0; i < QP; ++i) {
          const uint32_t w[4] = {cw[i].x, cw[i].y, cw[i].z, cw[i].w};
          uint32_t o[16];
          if (QUANT == 4) {
#pragma unroll
            for (int u = 0; u < 4; ++u) dequant_word(w[u], mw[i], &o[4 * u]);
          } else {
            dequant_group3(w[0], w[1], w[2], w[3], o);
          }
          if (ks + 2 < nst) fetch(ks + 2, i);              // on its way while the other passes are converted
#pragma unroll
          for (int u = 0; u < 4; ++u)                      // 32 tile rows on: 4096 bytes (the swizzle repeats every 8)
            asm volatile("st.shared.v4.u32 [%0], {%1,%2,%3,%4};" ::"r"(to[u] + 4096u * (uint32_t)i), "r"(o[4 * u]), "r"(o[4 * u + 1]), "r"(o[4 * u + 2]), "r"(o[4 * u + 3]) : "memory");
        }
        asm volatile("cp.async.wait_all;" ::: "memory");   // the staged rotary rows of this tile (key stream) have landed too
        fence_proxy_async();                               // the tensor core reads these stores
        mbar_arrive(BAR(bar_full + pr));                   // the pair is complete when all threads of the stream are done
        ++pairs;
        slot += 2;
        if (slot == RS) slot = 0;
      }
    };
    auto load_rows_q = [&](uint32_t (&gw)[QP]) {           // (less than 2^24 rows of at most 256 groups)
#pragma unroll
      for (int i = 0; i < QP; ++i) {
        const int p = pos_s[pb * kTile + (int)rq + 32 * i];
        gw[i] = (p < 0 ? 0u : (uint32_t)p) * (uint32_t)(r >> 5);
      }
    };
    auto load_rows = [&](uint32_t (&ro)[16]) {             // rows without a selected token read row 0 (weight 0)
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        const int p = pos_s[pb * kTile + (int)r8 + 8 * i];
        ro[i] = p < 0 ? 0u : (uint32_t)p;
      }
    };
    // One loop for both streams (one copy of the issue code).  The key stream also publishes the row positions and
    // the coarse rotary rows of every tile: thread t loads the positions of tile rows t, t + SPT, ..., one tile ahead;
    // the range check is made when the value is used, so that nobody waits for the load here.
    TileIter cur, nxt;
    iter_begin(nxt);
    bool have = iter_next(nxt, no_op, no_op);
    if (kstream && (dev.inject & XKV_INJECT_FUSED_NO_ROWS)) have = false;   // fault injection: no positions, no rows of A_k
    auto load_pos = [&](const TileIter& x, int row) {
      return (x.ti * kTile + row < x.cnt) ? sel_idx[x.prob * sc.k_cap + x.ti * kTile + row] : -1;
    };
    auto checked = [&](const TileIter& x, int row, int p) {
      if (x.ti * kTile + row < x.cnt && (p < 0 || p >= dev.T)) { atomicOr(dev.flags, XKV_FLAG_INDEX_RANGE); p = -1; }
      return p;
    };
    constexpr int PP = kTile / SPT;                        // positions per thread
    int pn[PP];
#pragma unroll
    for (int i = 0; i < PP; ++i) pn[i] = kstream && have ? load_pos(nxt, ts + SPT * i) : -1;
    while (ok && have) {
      cur = nxt;
      int pq[PP];
#pragma unroll
      for (int i = 0; i < PP; ++i) pq[i] = kstream ? checked(cur, ts + SPT * i, pn[i]) : -1;
      have = iter_next(nxt, no_op, no_op);
      if (kstream) {
        if (have) {
#pragma unroll
          for (int i = 0; i < PP; ++i) pn[i] = load_pos(nxt, ts + SPT * i);
        }
        const int buf = it & 1;
        // the key epilogue must be done with this buffer's rotary rows (tile it-2), and the value stream with
        // the positions of tile it-4
        if (!wait_bar(ctx, BAR(bl.rfree + buf), (uint32_t)(((it >> 1) & 1) ^ 1), ps + 1)) { ok = false; break; }
        if (it >= 4 && !wait_bar(ctx, BAR(bl.vfree + pb), (uint32_t)(((it >> 2) & 1) ^ 1), ps + 1)) { ok = false; break; }
#pragma unroll
        for (int i = 0; i < PP; ++i) pos_s[pb * kTile + ts + SPT * i] = pq[i];
        if (rope_smem) {
          // rows 8a..8a+7 of the tile are usually the eight positions of one coarse rotary row (a landmark chunk): stage it once.
          // Warp pw handles the 32-row blocks pw, pw + PW / 2, ... (lane = row inside the block).
#pragma unroll
          for (int hb = 0; hb < PP; ++hb) {
            const int blk = pw + (PW / 2) * hb, p = pq[hb];
            const int hidx = p < 0 ? -1 : (p >> 3);
            int gmax = hidx;
            gmax = max(gmax, __shfl_xor_sync(0xffffffffu, gmax, 1));
            gmax = max(gmax, __shfl_xor_sync(0xffffffffu, gmax, 2));
            gmax = max(gmax, __shfl_xor_sync(0xffffffffu, gmax, 4));
            const bool aligned = __all_sync(0xffffffffu, p < 0 || hidx == gmax);
            const bool in_order = __all_sync(0xffffffffu, p < 0 || (p & 7) == (lane & 7));
            if (lane == 0) algn_s[buf * 4 + blk] = aligned ? in_order ? 1 : 2 : 0;
            if (aligned) {
#pragma unroll
              for (int a = 0; a < 4; ++a) {
                const int gm = __shfl_sync(0xffffffffu, gmax, a * 8);
                if (lane < UN) {
                  cp_async16(smem_u32(hi_s + (size_t)(buf * 16 + blk * 4 + a) * UN + lane),
                             dev.rope_hi + (size_t)(gm < 0 ? 0 : gm) * UN + lane, 16u);
                }
              }
            }
          }
        }
        // publish the row positions of the tile (to both streams and to the key epilogue)
        mbar_arrive(BAR(bl.posfull + pb));
      }
      if (!wait_bar(ctx, BAR(bl.posfull + pb), (uint32_t)((it >> 2) & 1), ps + 2)) { ok = false; break; }
      if constexpr (QUANT != 0) {
        uint32_t gw[QP];
        load_rows_q(gw);
        if (!kstream) mbar_arrive(BAR(bl.vfree + pb));     // this thread is done with the position buffer
        issue_phase_q(gw, cur.b);
      } else {
        uint32_t ro[16];
        load_rows(ro);
        if (!kstream) mbar_arrive(BAR(bl.vfree + pb));     // this thread is done with the position buffer
        issue_phase(ro, cur.b);
      }
      ++it;
      if (++pb == 4) pb = 0;
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    if (ctx.prof && (warp == 8 || warp == 8 + PW / 2) && lane == 0) {
      ctx.prof[ps] = (unsigned long long)(clock64() - role_t0);
      if (warp == 8) ctx.prof[4] = (unsigned long long)it;
    }
  } else if (warp == kWarpK || warp == kWarpV) {
    // =============================== MMA issue: one warp the key phases, one the value phases ===============
    // Two issuing threads, each walking its own ring (one thread spends 70-130 cycles per tcgen05.mma and about
    // 235 per tcgen05.commit).
    const bool kside = warp == kWarpK;
    // The whole warp walks the loop, one elected lane issues.  The key side is a critical chain of the kernel (with four
    // waits per slot pair, of 10.0 k cycles a tile it waited for data in 2.1 k and issued in 3.8 k; the rest were its own
    // instructions between the two; of 7.6 k now 1.9, 3.0 and 2.6), so a slot pair costs it one wait (gathered rows and B_k
    // slabs arrive on one barrier), and branches outside the issue are taken on a vote, so that the compiler may keep the
    // descriptors in uniform registers, where the tensor-core instructions take them from.  The kernel alone: 131072 rows,
    // budget 4096, rank 512 45.1 -> 41.7 us; 65536 rows, budget 16384, rank 1024 255.8 -> 239.7; eight heads, rank 256 75.1
    // -> 70.2; one tile per CTA 18.1 -> 17.2.  (Of the first a step shows little: kernel and merge back to back over eight
    // windows 45.4 -> 41.2 us with the order of the tiles, behind the selections 76.8 -> 75.9.)
    constexpr uint32_t idesc_k = idesc_bf16_f32(128, 128);                     // keys: both operands K-major
    constexpr uint32_t idesc_v = idesc_bf16_f32(128, 16) | (1u << 15);         // values: A is read along its rows (MN-major)
    const int ps = kside ? 8 : 40;
    const long long role_t0 = clock64();
    // This warp is the only consumer of its ring's `full` barriers and sees every phase of them in order, so one
    // parity bit per pair is enough.
    uint32_t pr = 0, seen = 0;
    // descriptors differ between slots only in the start-address field (units of 16 bytes)
    const uint64_t desc_hi = smem_desc_sw128(0, 0) & 0xFFFFFFFF00000000ull;
    constexpr uint32_t kSlab16 = kSlabBytes >> 4;
    const uint32_t rows_lo0 = (uint32_t)(smem_desc_sw128(base, 0) & 0xFFFFFFFFull);
    const uint32_t b_lo0 = (uint32_t)(smem_desc_sw128(bring, 0) & 0xFFFFFFFFull);
    // value phase: A = two adjacent row slabs of the value ring read transposed (64 rank columns each, 16384
    // bytes apart), rows advance in 8-row groups of 1024 bytes; B = the weights of 16 heads x 16 rows
    const uint32_t rows_t_lo0 = (((rows_lo0 & 0xFFFFu) + (uint32_t)SK * kSlab16) & 0xFFFFu) | (kSlab16 << 16);
    const uint32_t p_lo0 = (uint32_t)(smem_desc_sw128(P_addr, 0) & 0xFFFFFFFFull);
    auto wait_all = [&](uint32_t bar, uint32_t parity, int word) {
      return __all_sync(0xffffffffu, wait_bar(ctx, bar, parity, word)) != 0;
    };
    // Rows that were copied asynchronously are writes of the generic proxy, and their threads go on without waiting for them:
    // the fence towards the tensor core's reads is this warp's, behind the wait.  (The quantised streams store their rows
    // and fence themselves, before they arrive.)  It costs 0.2 to 0.9 % of a step: 131072 rows, budget 4096, 78.3 -> 78.7 us;
    // 65536 rows, budget 16384, 318.7 -> 319.6; 32768 rows by layer 113.4 -> 114.1.
    auto wait_rows = [&](uint32_t bar, uint32_t parity, int word) {
      const bool landed = wait_all(bar, parity, word);
      if constexpr (QUANT == 0) fence_proxy_async();
      tc_fence_after();
      return landed;
    };
    int it = 0;
    bool ok = true;
    TileIter cur;
    iter_begin(cur);
    while (ok && __all_sync(0xffffffffu, iter_next(cur, no_op, no_op))) {
      const int buf = it & 1;
      const uint32_t par = (uint32_t)((it >> 1) & 1);
      if (kside) {
        // ---- keys: K_hat = A_k[S] B_k
        const int last_kk = (((dev.r_k - 1) & 63) >> 4) + 1;    // 16-column steps in the last real slab
        const uint32_t acc = tmem + (uint32_t)(buf * 128);
        if (!wait_all(BAR(bl.kempty + buf), par ^ 1u, ps + 1)) { ok = false; break; }
        tc_fence_after();
#pragma unroll 1
        for (int ks = 0; ks < nst_k; ks += 2) {
          // one ring-slot pair per iteration: rows and B slabs of both slots, then all steps at once
          if (!wait_rows(BAR(bl.full) + 8u * pr, (seen >> pr) & 1u, ps + 3)) { ok = false; break; }
          seen ^= 1u << pr;
          const long long i0 = ctx.prof ? clock64() : 0;
          const uint64_t a_desc = desc_hi | (rows_lo0 + pr * (2u * kSlab16));
          const uint64_t b_desc = desc_hi | (b_lo0 + pr * (2u * kSlab16));
          const int nkk0 = (ks == nks_k - 1) ? last_kk : 4;
          const int nkk1 = (ks + 1 >= nks_k) ? 0 : ((ks + 1 == nks_k - 1) ? last_kk : 4);   // the second slab of the last pair may be padding
          if (elect_one()) {
            tc_mma_bf16(acc, a_desc, b_desc, idesc_k, ks ? 1u : 0u);
#pragma unroll
            for (int kk = 1; kk < 4; ++kk) {
              if (kk < nkk0) tc_mma_bf16(acc, a_desc + 2u * kk, b_desc + 2u * kk, idesc_k, 1u);   // +32 bytes per step
            }
#pragma unroll
            for (int kk = 0; kk < 4; ++kk) {
              if (kk < nkk1) tc_mma_bf16(acc, a_desc + kSlab16 + 2u * kk, b_desc + kSlab16 + 2u * kk, idesc_k, 1u);
            }
            tc_commit(BAR(bl.emptyk) + 8u * pr);       // releases both slots of the pair (and their B slabs)
            if (ks + 2 >= nst_k) tc_commit(BAR(bl.kfull + buf));
          }
          __syncwarp();
          if (ctx.prof && lane == 0) atomicAdd(ctx.prof + ps + 4, (unsigned long long)(clock64() - i0));
          if (++pr == SK / 2) pr = 0;
        }
      } else {
        // ---- values: W += A_v[S]^T P^T, one accumulator of 16 columns per 128 rank columns
        if (!wait_all(BAR(bl.wempty + buf), par ^ 1u, ps + 1)) { ok = false; break; }
        if (!wait_all(BAR(bl.pfull + buf), par, ps + 5)) { ok = false; break; }
        tc_fence_after();
        const uint32_t accw = tmem + 256u + (uint32_t)(buf * 128);
        const uint64_t p_desc = desc_hi | (p_lo0 + (uint32_t)buf * (kPBytes >> 4));
#pragma unroll 1
        for (int ks = 0; ks < nst_v; ks += 2) {
          if (!wait_rows(BAR(bl.fullv) + 8u * pr, (seen >> pr) & 1u, ps + 3)) { ok = false; break; }
          seen ^= 1u << pr;
          const long long i0 = ctx.prof ? clock64() : 0;
          const uint64_t a_desc = desc_hi | (rows_t_lo0 + pr * (2u * kSlab16));
          const uint32_t acc = accw + (uint32_t)(ks >> 1) * 16u;
          if (elect_one()) {
#pragma unroll
            for (int kk = 0; kk < 8; ++kk)   // 16 tile rows per step: 2048 bytes down the slab, 32 bytes along P
              tc_mma_bf16(acc, a_desc + (uint32_t)kk * (2048u >> 4), p_desc + (uint32_t)(kk >> 2) * (2048u >> 4) + (uint32_t)(kk & 3) * 2u,
                          idesc_v, kk ? 1u : 0u);
            tc_commit(BAR(bl.emptyv) + 8u * pr);
            if (ks + 2 >= nst_v) tc_commit(BAR(bl.wfull + buf));
          }
          __syncwarp();
          if (ctx.prof && lane == 0) atomicAdd(ctx.prof + ps + 4, (unsigned long long)(clock64() - i0));
          if (++pr == SV / 2) pr = 0;
        }
      }
      ++it;
    }
    if (ctx.prof && lane == 0) ctx.prof[ps] = (unsigned long long)(clock64() - role_t0);
    if (!ok && elect_one()) {          // (the lane that issued)
      // giving up: the tensor-core operations this thread has issued may still be running and the CTA is about to
      // free its tensor memory; wait (again with a limit) until they have retired
      const uint32_t db = BAR(bl.drain + (kside ? 0 : 1));
      tc_commit(db);
      for (uint32_t i = 0; i < (1u << 22); ++i) if (mbar_try_wait(db, 0)) break;
    }
    __syncwarp();
  } else if (warp == kWarpB) {
    // =============================== B_k slab loader (TMA) ===============================
    // The slabs of a slot pair of the key ring go to the same pair of their own ring, are released with it and arrive on its
    // barrier: the loader walks the pairs as the key stream's producers do.
    // fault injection (tests of the give-up path): the slabs are never loaded, so the key-phase warp's wait for
    // them runs into its limit and the CTA winds down
    const bool no_b = (dev.inject & XKV_INJECT_FUSED_NO_B) != 0u;
    uint32_t pr = 0, used = 0, rel_par = 0;   // per slot pair: filled before; parity of the release to wait for next
    bool ok = true;
    TileIter cur;
    iter_begin(cur);
    while (ok && lane == 0 && iter_next(cur, no_op, no_op)) {
      const int head_row = (int)((((size_t)cur.b * dev.G + cur.l) * dev.H_kv + cur.g) * kDP);
#pragma unroll 1
      for (int ks = 0; ks < nst_k; ks += 2) {
        const uint32_t bit = 1u << pr;
        if (used & bit) {
          if (!wait_bar(ctx, BAR(bl.emptyk) + 8u * pr, (rel_par >> pr) & 1u, 17)) { ok = false; break; }
          rel_par ^= bit;
        }
        used |= bit;
        if (!no_b) {
          const uint32_t dst = bring + pr * (2u * kSlabBytes), bar = BAR(bl.full) + 8u * pr;
          const bool second = ks + 1 < nks_k;          // the second slab of the last pair may be padding: not multiplied
          mbar_expect_tx(bar, second ? 2u * kSlabBytes : (uint32_t)kSlabBytes);
          tma_load_2d(dst, &bk_map, ks * 64, head_row, bar);
          if (second) tma_load_2d(dst + kSlabBytes, &bk_map, ks * 64 + 64, head_row, bar);
          ++pairs;
        }
        if (++pr == SK / 2) pr = 0;
      }
    }
    if (lane == 0) walk_s->loaded = pairs;
  } else if (warp < 4) {
    // =============================== key epilogue: rope, logits, softmax statistics, weights ===============================
    // tile row whose softmax terms this thread works on (quad_logits leaves the logits there)
    const int quad_t = lane & 3, quad_g = lane >> 2;
    const int j = warp * 32 + quad_t * 8 + quad_g;
    const uint32_t lane_base = (uint32_t)(warp * 32) << 16;
    const float scale2 = dev.att_scale * kLog2e;
    const int rmask = (1 << dev.rope_shift) - 1;
    float m_run[NR], l_thr[NR];
    int it = 0;
    bool ok = true;
    uint32_t grp_par = 0;
    const int ps = warp == 0 ? 24 : -1000;
    int pbuf = 0;                                       // position buffer of the tile (four in rotation)
    const long long role_t0 = clock64();
    // where this row's weights go in the bf16 operand tile: [row block j/64][head][64 rows], 128-byte swizzle
    const uint32_t p_off = (uint32_t)(j >> 6) * 2048u + (uint32_t)(j & 7) * 2u;
    const uint32_t p_unit = (uint32_t)((j & 63) >> 3);
    // barrier among the 128 threads of this role, with the same bounded wait as every other wait
    auto group_sync = [&]() {
      mbar_arrive(BAR(bl.grp));
      if (!wait_bar(ctx, BAR(bl.grp), grp_par, ps + 3)) ok = false;
      grp_par ^= 1u;
    };
    TileIter cur;
    iter_begin(cur);
    auto flush = [&](int py) {   // end of a segment: write (m, l) of every head to the problem's partial slot
      float tot[NR];
#pragma unroll
      for (int h = 0; h < NR; ++h) {
        float v = l_thr[h];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        tot[h] = v;
      }
      group_sync();                                     // red_s[0] is free (last tile's readers are done)
      if (lane == 0) {
#pragma unroll
        for (int h = 0; h < NR; ++h) red_s[warp * NR + h] = tot[h];
      }
      group_sync();
      if (j < n_rep) {
        float* part = part_of(py, cur.prob) + (size_t)j * (dev.r_v + 2) + dev.r_v;
        float ls = 0.0f, mm = -INFINITY;
#pragma unroll
        for (int h = 0; h < NR; ++h) {
          if (h == j) { ls = red_s[h] + red_s[NR + h] + red_s[2 * NR + h] + red_s[3 * NR + h]; mm = m_run[h]; }
        }
        part[0] = mm;
        part[1] = ls;
      }
    };
    auto on_leave = [&]() { flush(cur.py); };
    auto on_enter = [&]() {
#pragma unroll
      for (int h = 0; h < NR; ++h) { m_run[h] = -INFINITY; l_thr[h] = 0.0f; }
      const __nv_bfloat16* qg = q + (((long long)cur.l * dev.batch + cur.b) * dev.H_q + (long long)cur.g * n_rep) * DH;
      // 16-byte pieces, all of a thread's loads issued before the first is used (heads beyond n_rep are zero)
      {
        constexpr int kPieces = NR * DH / 8, kPer = (kPieces + 127) / 128;
        const uint4* qv = reinterpret_cast<const uint4*>(qg);
        uint4 u[kPer];
#pragma unroll
        for (int i = 0; i < kPer; ++i) {
          const int pc = j + 128 * i;
          u[i] = (pc < kPieces && pc * 8 < n_rep * DH) ? __ldg(qv + pc) : make_uint4(0u, 0u, 0u, 0u);
        }
#pragma unroll
        for (int i = 0; i < kPer; ++i) {
          const int pc = j + 128 * i;
          if (pc < kPieces) {
            // eight dimensions: half of four units
            const int h = pc / (DH / 8), m = pc % (DH / 8);
            float* to = q_s + h * DH + (m % (HALF / 8)) * 16 + (m / (HALF / 8)) * 2;
            const uint32_t w[4] = {u[i].x, u[i].y, u[i].z, u[i].w};
#pragma unroll
            for (int e = 0; e < 4; ++e)
              *reinterpret_cast<float2*>(to + 4 * e) = make_float2(__uint_as_float(w[e] << 16), __uint_as_float(w[e] & 0xffff0000u));
          }
        }
      }
      group_sync();
    };
    while (ok && iter_next(cur, on_leave, on_enter)) {
      const int buf = it & 1;
      const uint32_t par = (uint32_t)((it >> 1) & 1);
      if (!wait_bar(ctx, BAR(bl.posfull + pbuf), (uint32_t)((it >> 2) & 1), ps + 1)) { ok = false; break; }   // positions published
      if (!wait_bar(ctx, BAR(bl.kfull + buf), par, ps + 2)) { ok = false; break; }
      tc_fence_after();
      const int pos = pos_s[pbuf * kTile + j], own = pos_s[pbuf * kTile + tid];   // own: of the row in this thread's TMEM lane
      if (++pbuf == 4) pbuf = 0;
      float z[NR];
      const uint32_t acc = tmem + lane_base + (uint32_t)(buf * 128);
      const int staged = rope_smem ? algn_s[buf * 4 + warp] : 0;      // 1: whole chunks in order, 2: in another order
      bool by_row = staged != 1;
      if (!by_row) {
        quad_logits<DH, NR, MMA>(acc, reinterpret_cast<const ulonglong2*>(hi_s + (buf * 16 + warp * 4) * UN),
                                 reinterpret_cast<const ulonglong2*>(lo_s + quad_g * UN), lo_swz(quad_g),
                                 reinterpret_cast<const uint4*>(q_s), lane, z);
        if constexpr (MMA) {
          // an infinite key element has no upper part and rest: such a row's logits come out as NaN there, also one that is
          // minus infinity and takes no part in the softmax
          bool nan = false;
#pragma unroll
          for (int h = 0; h < NR; ++h) nan |= h < n_rep && z[h] != z[h];
          by_row = __any_sync(0xffffffffu, nan && pos >= 0);
        }
      }
      if (by_row) {
        const int pp = own < 0 ? 0 : own;
        const ulonglong2* qv = reinterpret_cast<const ulonglong2*>(q_s);
        const LogitsOut<NR> o =
            staged ? key_logits_rows<DH, NR, QUANT, kStagedTables>(acc, smem_u32(hi_s + (buf * 16 + (tid >> 3)) * UN),
                                                               smem_u32(lo_s + (pp & 7) * UN), lo_swz(pp & 7), qv)
            : dev.use_rope ? key_logits_rows<DH, NR, QUANT, kHandleTables>(acc, (u64)(dev.rope_hi + (size_t)(pp >> dev.rope_shift) * UN),
                                                                       (u64)(dev.rope_lo + (size_t)(pp & rmask) * UN), 0, qv)
                           : key_logits_rows<DH, NR, QUANT, kNoTables>(acc, 0, 0, 0, qv);
#pragma unroll
        for (int h = 0; h < NR; ++h) z[h] = __shfl_sync(0xffffffffu, o.z[h], quad_t * 8 + quad_g);
      }
      tc_fence_before();
      mbar_arrive(BAR(bl.kempty + buf));                // accumulator may be overwritten
      mbar_arrive(BAR(bl.rfree + buf));                 // positions and rotary rows of this tile are consumed
      // tile max per head over the 128 rows
      // (one redux.sync per head on the order-preserving integer image of the float: exact, and a fraction of
      // the code of a shuffle tree)
      float tmax[NR];
#pragma unroll
      for (int h = 0; h < NR; ++h) {
        z[h] = pos < 0 ? -INFINITY : z[h] * scale2;
        int zi = __float_as_int(z[h]);
        zi ^= (zi >> 31) & 0x7fffffff;
        int mi = __reduce_max_sync(0xffffffffu, zi);
        mi ^= (mi >> 31) & 0x7fffffff;
        tmax[h] = __int_as_float(mi);
      }
      float* red = red_s + (it & 1) * 4 * NR;
      if (lane == 0) {
#pragma unroll
        for (int h = 0; h < NR; ++h) red[h * 4 + warp] = tmax[h];   // [head][warp]: one 16-byte load per head below
      }
      group_sync();
      if (!ok) break;
      // the weights buffer and the rescale factors of tile it-2 must have been consumed
      if (!wait_bar(ctx, BAR(bl.wempty + buf), par ^ 1u, ps + 4)) { ok = false; break; }
      uint8_t* Pw = P_gen + buf * kPBytes + p_off;
#pragma unroll
      for (int h = 0; h < NR; ++h) {
        const float4 t4 = *reinterpret_cast<const float4*>(red + h * 4);
        const float tm = fmaxf(fmaxf(t4.x, t4.y), fmaxf(t4.z, t4.w));
        const float m_new = fmaxf(m_run[h], tm);
        const float alpha = (m_run[h] == -INFINITY) ? 0.0f : ex2_approx(m_run[h] - m_new);
        const float p = (m_new == -INFINITY) ? 0.0f : ex2_approx(z[h] - m_new);
        const __nv_bfloat16 pb = __float2bfloat16(p);
        l_thr[h] = l_thr[h] * alpha + __bfloat162float(pb);   // the denominator sums the weights as they are used
        m_run[h] = m_new;
        if (h < n_rep) *reinterpret_cast<__nv_bfloat16*>(Pw + h * 128 + ((p_unit ^ (uint32_t)(h & 7)) << 4)) = pb;
        if (j == h) alpha_s[buf * NR + h] = alpha;
      }
      fence_proxy_async();                              // the weights are read by the tensor core
      mbar_arrive(BAR(bl.pfull + buf));
      ++it;
    }
    if (ok && cur.py >= 0) flush(cur.py);
    if (ctx.prof && j == 0) ctx.prof[24] = (unsigned long long)(clock64() - role_t0);
  } else {
    // =============================== value epilogue: running W = W * alpha + W_tile ===============================
    const int mm = tid - 128;                           // rank column inside a 128-column block = TMEM lane
    const uint32_t lane_base = (uint32_t)((warp - 4) * 32) << 16;
    const int nblk = (dev.r_v + 127) >> 7;
    float w[WB][NR];
    const int ps = warp == 4 ? 32 : -1000;
    const long long role_t0 = clock64();
    int it = 0;
    bool ok = true;
    TileIter cur;
    iter_begin(cur);
    auto flush = [&](int py) {
      float* part = part_of(py, cur.prob);
#pragma unroll
      for (int bk = 0; bk < WB; ++bk) {
        const int col = bk * 128 + mm;
        if (bk < nblk && col < dev.r_v) {
#pragma unroll
          for (int h = 0; h < NR; ++h) if (h < n_rep) part[(size_t)h * (dev.r_v + 2) + col] = w[bk][h];
        }
      }
    };
    auto on_leave = [&]() { flush(cur.py); };
    auto on_enter = [&]() {
#pragma unroll
      for (int bk = 0; bk < WB; ++bk)
#pragma unroll
        for (int h = 0; h < NR; ++h) w[bk][h] = 0.0f;
    };
    while (ok && iter_next(cur, on_leave, on_enter)) {
      const int buf = it & 1;
      const uint32_t par = (uint32_t)((it >> 1) & 1);
      if (!wait_bar(ctx, BAR(bl.wfull + buf), par, ps + 1)) { ok = false; break; }
      tc_fence_after();
      float al[NR];
#pragma unroll
      for (int h = 0; h < NR; ++h) al[h] = alpha_s[buf * NR + h];
      const uint32_t acc = tmem + lane_base + 256u + (uint32_t)(buf * 128);
#pragma unroll
      for (int bk = 0; bk < WB; ++bk) {
        if (bk < nblk) {
          float v[NR];
          tmem_ld<NR>(acc + (uint32_t)(bk * 16), v);
          tc_wait_ld();
#pragma unroll
          for (int h = 0; h < NR; ++h) w[bk][h] = fmaf(w[bk][h], al[h], v[h]);
        }
      }
      tc_fence_before();
      mbar_arrive(BAR(bl.wempty + buf));
      ++it;
    }
    if (ok && cur.py >= 0) flush(cur.py);
    if (ctx.prof && mm == 0) ctx.prof[32] = (unsigned long long)(clock64() - role_t0);
  }

  // wind down: nothing of this CTA may still touch shared or tensor memory
  asm volatile("cp.async.wait_all;" ::: "memory");
  tc_fence_before();
  __syncthreads();
  if (warp == kWarpK) {
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
  if (*abort_flag) {
    // Given up: slabs of B_k may still be on their way into this CTA's shared memory, which the next CTA on the SM would
    // inherit.  They arrive on barriers that count the key stream's threads too: those make up the arrivals that they owe
    // the pairs requested, so that a pair's phase ends with its last byte, and the loader stays (again with a limit) for it.
    const uint32_t loaded = walk_s->loaded;
    if (warp >= 8 && warp < 8 + PW / 2) {
      for (uint32_t n = pairs; n < loaded; ++n) mbar_arrive(BAR(bl.full) + 8u * (n % (SK / 2)));
    } else if (warp == kWarpB && lane == 0) {
      for (uint32_t n = loaded > SK / 2 ? loaded - SK / 2 : 0u; n < loaded; ++n)
        for (uint32_t i = 0; i < (1u << 22); ++i) if (mbar_try_wait(BAR(bl.full) + 8u * (n % (SK / 2)), (n / (SK / 2)) & 1u)) break;
    }
  }
}

// Partials of a problem -> out, lse.  grid.x = problems * n_rep, 1024 threads.  m is in log2 units.
// W_h = sum_seg 2^(m_seg - M) W_seg[h], L = sum_seg 2^(m_seg - M) l_seg, then
// out_h[d] = (1/L) sum_m W_h[m] B_v[m][g*d_h + d]   (Eq. 3 applied once to the weighted sum of basis rows).
// DH/8 threads read one 16-byte piece each of a B_v row; 1024/(DH/8) rows are in flight per pass.
constexpr int kMergeThreads = 1024;
constexpr int kMergeMaxSeg = 160;                     // a problem never has more segments than there are CTAs + 1
template <int DH>
__global__ void __launch_bounds__(kMergeThreads)
merge_segments_kernel(GroupDev dev, Sched sc, TailParts tail, __nv_bfloat16* __restrict__ out, float* __restrict__ lse) {
  extern __shared__ float m_s[];                      // [r_v] weights-times-basis, then [rows per pass][DH] partial sums
  __shared__ float wgt_s[kMergeMaxSeg];
  __shared__ float twgt_s[kTailMaxSplit];             // weights of the partial results over the uncompressed tail
  __shared__ float ML_s[2];
  constexpr int TPR = DH / 8, RPP = kMergeThreads / TPR;
  const int n_rep = dev.n_rep, r = dev.r_v;
  float* w_s = m_s;
  float* red = m_s + ((r + 3) & ~3);
  const int tid = threadIdx.x;
  const int h = blockIdx.x % n_rep, py = blockIdx.x / n_rep;
  const int per_layer = dev.batch * dev.H_kv;
  const int g = py % dev.H_kv, b = (py / dev.H_kv) % dev.batch, l = sc.l0 + py / per_layer;
  const long long prob = ((long long)l * dev.batch + b) * dev.H_kv + g;
  const int first = py * sc.tpp;
  const int c0 = cta_of_tile(sc, first), c1 = cta_of_tile(sc, first + sc.tpp - 1);
  const int nseg = min(c1 - c0 + 1, kMergeMaxSeg);
  const size_t stride = (size_t)n_rep * (r + 2);
  // the B_v pieces do not depend on the partials: start those loads before anything else
  const int rg = tid / TPR, dg = tid % TPR;
  const size_t ld = (size_t)dev.H_kv * DH;
  const __nv_bfloat16* Bv = dev.B_v + (((size_t)b * dev.G + l) * r) * ld + (size_t)g * DH + dg * 8;
  constexpr int kPre = 8;                             // rows of B_v held in registers per thread
  uint4 pre[kPre];
#pragma unroll
  for (int i = 0; i < kPre; ++i) {
    const int m = rg + i * RPP;
    pre[i] = m < r ? *reinterpret_cast<const uint4*>(Bv + (size_t)m * ld) : make_uint4(0, 0, 0, 0);
  }
  grid_dependency_wait();                             // the partials come from the kernel launched before this one
  grid_dependency_launch();                           // the next kernel of the stream may start its own set-up
  const float* part = dev.part + ((size_t)prob * sc.n_slots) * stride + (size_t)h * (r + 2);
  const int nts = tail.part ? min(tail.n_split, kTailMaxSplit) : 0;
  const size_t tstride = (size_t)n_rep * (DH + 2);
  const float* tpart = tail.part ? tail.part + ((size_t)py * tail.n_split) * tstride + (size_t)h * (DH + 2) : nullptr;
  // this thread's column of the first segments' partial sums: fetched together with the statistics below, so
  // that the merge costs one round trip to L2 instead of two
  constexpr int kSegPre = 8;
  static_assert(kMaxBlocks * 128 <= kMergeThreads, "one rank column per thread");
  float pv[kSegPre];
#pragma unroll
  for (int s = 0; s < kSegPre; ++s) pv[s] = (s < nseg && tid < r) ? __ldcg(part + s * stride + tid) : 0.0f;
  // and its share of the first partial results over the uncompressed tail (which are already in output space): with them
  // and their statistics in the same batch a step with a 1500-row tail takes 187.7 us instead of 193.4
  constexpr int FOLD = kMergeThreads / DH;            // 8 (d_h = 128) or 16 (d_h = 64) threads per column
  constexpr int kTailPre = 2;
  const int od = tid % DH, of = tid / DH;
  float tv[kTailPre];
#pragma unroll
  for (int i = 0; i < kTailPre; ++i) tv[i] = of + i * FOLD < nts ? __ldcg(tpart + (of + i * FOLD) * tstride + od) : 0.0f;
  if (tid < 32) {                                     // one warp: maxima, weights of the segments, denominator
    // maxima and denominators of this lane's segments in one batch of loads
    constexpr int kPer = (kMergeMaxSeg + 31) / 32;
    float sm[kPer], sl[kPer];
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
      const int s = tid + 32 * i;
      sm[i] = s < nseg ? __ldcg(part + s * stride + r) : -INFINITY;
      sl[i] = s < nseg ? __ldcg(part + s * stride + r + 1) : 0.0f;
    }
    const float tm = tid < nts ? __ldcg(tpart + tid * tstride + DH) : -INFINITY;
    const float tl = tid < nts ? __ldcg(tpart + tid * tstride + DH + 1) : 0.0f;
    float mx = tm;
#pragma unroll
    for (int i = 0; i < kPer; ++i) mx = fmaxf(mx, sm[i]);
    for (int s = tid + 32; s < nts; s += 32) mx = fmaxf(mx, tpart[s * tstride + DH]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    float Ls = 0.0f;
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
      const int s = tid + 32 * i;
      if (s < nseg) {
        const float w = (sm[i] == -INFINITY || mx == -INFINITY) ? 0.0f : exp2f(sm[i] - mx);
        wgt_s[s] = w;
        Ls += w * sl[i];
      }
    }
    if (tid < nts) {
      const float w = (tm == -INFINITY || mx == -INFINITY) ? 0.0f : exp2f(tm - mx);
      twgt_s[tid] = w;
      Ls += w * tl;
    }
    for (int s = tid + 32; s < nts; s += 32) {
      const float ms = tpart[s * tstride + DH];
      const float w = (ms == -INFINITY || mx == -INFINITY) ? 0.0f : exp2f(ms - mx);
      twgt_s[s] = w;
      Ls += w * tpart[s * tstride + DH + 1];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) Ls += __shfl_xor_sync(0xffffffffu, Ls, o);
    if (tid == 0) { ML_s[0] = mx; ML_s[1] = Ls; }
  }
  __syncthreads();
  if (tid < r) {                                      // r <= kMergeThreads
    float acc = 0.0f;
#pragma unroll
    for (int s = 0; s < kSegPre; ++s) if (s < nseg) acc = fmaf(wgt_s[s], pv[s], acc);
    for (int s = kSegPre; s < nseg; ++s) acc = fmaf(wgt_s[s], part[s * stride + tid], acc);
    w_s[tid] = acc;
  }
  __syncthreads();
  float acc[8];
#pragma unroll
  for (int e = 0; e < 8; ++e) acc[e] = 0.0f;
  auto add_row = [&](const uint4& v, float w) {
    const uint32_t u[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      acc[2 * e] = fmaf(w, __uint_as_float(u[e] << 16), acc[2 * e]);
      acc[2 * e + 1] = fmaf(w, __uint_as_float(u[e] & 0xffff0000u), acc[2 * e + 1]);
    }
  };
#pragma unroll
  for (int i = 0; i < kPre; ++i) {
    const int m = rg + i * RPP;
    if (m < r) add_row(pre[i], w_s[m]);
  }
#pragma unroll 4
  for (int m = rg + kPre * RPP; m < r; m += RPP) add_row(*reinterpret_cast<const uint4*>(Bv + (size_t)m * ld), w_s[m]);
#pragma unroll
  for (int e = 0; e < 8; ++e) red[rg * DH + dg * 8 + e] = acc[e];
  __syncthreads();
  // two-level sum over the row groups: 1024 threads fold RPP partials to 8 per column, then DH threads finish
  {
    float o = 0.0f;
#pragma unroll 4
    for (int i = of; i < RPP; i += FOLD) o += red[i * DH + od];
#pragma unroll
    for (int i = 0; i < kTailPre; ++i) if (of + i * FOLD < nts) o = fmaf(twgt_s[of + i * FOLD], tv[i], o);
#pragma unroll 4
    for (int s = of + kTailPre * FOLD; s < nts; s += FOLD) o = fmaf(twgt_s[s], tpart[s * tstride + od], o);
    __syncthreads();
    red[of * DH + od] = o;
  }
  __syncthreads();
  if (tid < DH) {
    float o = 0.0f;
#pragma unroll
    for (int f = 0; f < FOLD; ++f) o += red[f * DH + tid];
    const float M = ML_s[0], L = ML_s[1];
    const long long qh = ((long long)l * dev.batch + b) * dev.H_q + (long long)g * n_rep + h;
    out[qh * DH + tid] = __float2bfloat16(L > 0.0f ? o / L : 0.0f);
    if (lse && tid == 0) lse[qh] = L > 0.0f ? (M + log2f(L)) * kLn2 : -INFINITY;
  }
}

// The same merge for windows with many problems: one CTA per (problem, group of HG query heads), 512 threads.
// With one CTA per head a window of 128 problems x 7 heads is six waves of CTAs that each read the problem's B_v
// block again; here every B_v row a thread fetches serves all HG heads.  Same arithmetic per head as above; the
// sum over the rows of B_v is folded by one shuffle and one pass through shared memory.
constexpr int kMergeMultiThreads = 512;
template <int DH, int HG>
__global__ void __launch_bounds__(kMergeMultiThreads)
merge_segments_multi_kernel(GroupDev dev, Sched sc, TailParts tail, __nv_bfloat16* __restrict__ out, float* __restrict__ lse) {
  extern __shared__ float m_s[];                      // [HG][r4] weighted sums of basis rows, [HG][warps][DH] partial outputs
  __shared__ float wgt_s[HG][kMergeMaxSeg];
  __shared__ float twgt_s[HG][kTailMaxSplit];
  __shared__ float ML_s[HG][2];
  constexpr int TPR = DH / 8, RPP = kMergeMultiThreads / TPR, NW = kMergeMultiThreads / 32;
  const int n_rep = dev.n_rep, r = dev.r_v, r4 = (r + 3) & ~3;
  float* w_s = m_s;
  float* red = m_s + HG * r4;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int ngrp = (n_rep + HG - 1) / HG;
  const int h0 = (blockIdx.x % ngrp) * HG, py = blockIdx.x / ngrp;
  const int nh = min(HG, n_rep - h0);
  const int per_layer = dev.batch * dev.H_kv;
  const int g = py % dev.H_kv, b = (py / dev.H_kv) % dev.batch, l = sc.l0 + py / per_layer;
  const long long prob = ((long long)l * dev.batch + b) * dev.H_kv + g;
  const int first = py * sc.tpp;
  const int c0 = cta_of_tile(sc, first), c1 = cta_of_tile(sc, first + sc.tpp - 1);
  const int nseg = min(c1 - c0 + 1, kMergeMaxSeg);
  const size_t stride = (size_t)n_rep * (r + 2);
  const int rg = tid / TPR, dg = tid % TPR;
  const size_t ld = (size_t)dev.H_kv * DH;
  const __nv_bfloat16* Bv = dev.B_v + (((size_t)b * dev.G + l) * r) * ld + (size_t)g * DH + dg * 8;
  constexpr int kPre = HG <= 4 ? 8 : 4;               // rows of B_v requested before the partials are waited for
  uint4 pre[kPre];
#pragma unroll
  for (int i = 0; i < kPre; ++i) {
    const int m = rg + i * RPP;
    pre[i] = m < r ? *reinterpret_cast<const uint4*>(Bv + (size_t)m * ld) : make_uint4(0, 0, 0, 0);
  }
  grid_dependency_wait();
  grid_dependency_launch();
  const float* part0 = dev.part + ((size_t)prob * sc.n_slots) * stride + (size_t)h0 * (r + 2);
  const int nts = tail.part ? min(tail.n_split, kTailMaxSplit) : 0;
  const size_t tstride = (size_t)n_rep * (DH + 2);
  const float* tpart0 = tail.part ? tail.part + ((size_t)py * tail.n_split) * tstride + (size_t)h0 * (DH + 2) : nullptr;
  if (warp < nh) {                                    // warp h: maxima, weights of the segments, denominator of head h0 + h
    const float* part = part0 + (size_t)warp * (r + 2);
    const float* tpart = tpart0 ? tpart0 + (size_t)warp * (DH + 2) : nullptr;
    constexpr int kPer = (kMergeMaxSeg + 31) / 32;
    float sm[kPer], sl[kPer];
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
      const int sg = lane + 32 * i;
      sm[i] = sg < nseg ? __ldcg(part + sg * stride + r) : -INFINITY;
      sl[i] = sg < nseg ? __ldcg(part + sg * stride + r + 1) : 0.0f;
    }
    float mx = -INFINITY;
#pragma unroll
    for (int i = 0; i < kPer; ++i) mx = fmaxf(mx, sm[i]);
    for (int sg = lane; sg < nts; sg += 32) mx = fmaxf(mx, tpart[sg * tstride + DH]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    float Ls = 0.0f;
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
      const int sg = lane + 32 * i;
      if (sg < nseg) {
        const float w = (sm[i] == -INFINITY || mx == -INFINITY) ? 0.0f : exp2f(sm[i] - mx);
        wgt_s[warp][sg] = w;
        Ls += w * sl[i];
      }
    }
    for (int sg = lane; sg < nts; sg += 32) {
      const float ms = tpart[sg * tstride + DH];
      const float w = (ms == -INFINITY || mx == -INFINITY) ? 0.0f : exp2f(ms - mx);
      twgt_s[warp][sg] = w;
      Ls += w * tpart[sg * tstride + DH + 1];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) Ls += __shfl_xor_sync(0xffffffffu, Ls, o);
    if (lane == 0) { ML_s[warp][0] = mx; ML_s[warp][1] = Ls; }
  }
  __syncthreads();
  // weighted sums of the segments' partial sums, one rank column per thread and pass, segments in ascending order
  // (the loads of the first four segments of all heads are issued before the first of them is used: one trip to L2
  // per column, not one per head and segment)
  for (int col = tid; col < r; col += kMergeMultiThreads) {
    constexpr int kSegBatch = 4;
    float v[HG][kSegBatch];
#pragma unroll
    for (int h = 0; h < HG; ++h)
#pragma unroll
      for (int sg = 0; sg < kSegBatch; ++sg)
        v[h][sg] = (h < nh && sg < nseg) ? __ldcg(part0 + (size_t)h * (r + 2) + col + sg * stride) : 0.0f;
#pragma unroll
    for (int h = 0; h < HG; ++h) {
      if (h < nh) {
        const float* part = part0 + (size_t)h * (r + 2) + col;
        float acc = 0.0f;
#pragma unroll
        for (int sg = 0; sg < kSegBatch; ++sg) if (sg < nseg) acc = fmaf(wgt_s[h][sg], v[h][sg], acc);
        for (int sg = kSegBatch; sg < nseg; ++sg) acc = fmaf(wgt_s[h][sg], __ldcg(part + sg * stride), acc);
        w_s[h * r4 + col] = acc;
      }
    }
  }
  __syncthreads();
  float acc[HG][8];
#pragma unroll
  for (int h = 0; h < HG; ++h)
#pragma unroll
    for (int e = 0; e < 8; ++e) acc[h][e] = 0.0f;
  auto add_row = [&](const uint4& v, int m) {
    const uint32_t u[4] = {v.x, v.y, v.z, v.w};
    float x[8];
#pragma unroll
    for (int e = 0; e < 4; ++e) { x[2 * e] = __uint_as_float(u[e] << 16); x[2 * e + 1] = __uint_as_float(u[e] & 0xffff0000u); }
#pragma unroll
    for (int h = 0; h < HG; ++h) {
      const float w = h < nh ? w_s[h * r4 + m] : 0.0f;
#pragma unroll
      for (int e = 0; e < 8; ++e) acc[h][e] = fmaf(w, x[e], acc[h][e]);
    }
  };
#pragma unroll
  for (int i = 0; i < kPre; ++i) {
    const int m = rg + i * RPP;
    if (m < r) add_row(pre[i], m);
  }
  // the remaining rows four at a time, their loads issued together
  for (int m0 = rg + kPre * RPP; m0 < r; m0 += 4 * RPP) {
    uint4 nx[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int m = m0 + u * RPP;
      nx[u] = m < r ? *reinterpret_cast<const uint4*>(Bv + (size_t)m * ld) : make_uint4(0, 0, 0, 0);
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int m = m0 + u * RPP;
      if (m < r) add_row(nx[u], m);
    }
  }
  // a warp holds two row groups (lanes 0..15 and 16..31 with the same columns): fold them, then one partial per warp
#pragma unroll
  for (int h = 0; h < HG; ++h)
#pragma unroll
    for (int e = 0; e < 8; ++e) acc[h][e] += __shfl_xor_sync(0xffffffffu, acc[h][e], TPR);
  static_assert(TPR == 16 || TPR == 8, "row groups per warp");
  if constexpr (TPR == 8) {
#pragma unroll
    for (int h = 0; h < HG; ++h)
#pragma unroll
      for (int e = 0; e < 8; ++e) acc[h][e] += __shfl_xor_sync(0xffffffffu, acc[h][e], 16);
  }
  if (lane < TPR) {
#pragma unroll
    for (int h = 0; h < HG; ++h)
#pragma unroll
      for (int e = 0; e < 8; ++e) red[(h * NW + warp) * DH + lane * 8 + e] = acc[h][e];
  }
  __syncthreads();
  for (int o = tid; o < nh * DH; o += kMergeMultiThreads) {
    const int h = o / DH, d = o - h * DH;
    float v = 0.0f;
#pragma unroll
    for (int w = 0; w < NW; ++w) v += red[(h * NW + w) * DH + d];
    if (tpart0) {
      const float* tpart = tpart0 + (size_t)h * (DH + 2);
      for (int sg = 0; sg < nts; ++sg) v = fmaf(twgt_s[h][sg], tpart[sg * tstride + d], v);
    }
    const float M = ML_s[h][0], L = ML_s[h][1];
    const long long qh = ((long long)l * dev.batch + b) * dev.H_q + (long long)g * n_rep + h0 + h;
    out[qh * DH + d] = __float2bfloat16(L > 0.0f ? v / L : 0.0f);
    if (lse && d == 0) lse[qh] = L > 0.0f ? (M + log2f(L)) * kLn2 : -INFINITY;
  }
}

template <int DH, int NR>
constexpr size_t fused_smem_bytes() {
  return 1024 + (size_t)(2 * kKeySlots + value_slots<DH, NR>()) * kSlabBytes + misc_smem_bytes<DH, NR>();
}

template <int DH, int NR, int WB>
cudaError_t launch_fused_t(const xkv_group* grp, int l0, int l1, const __nv_bfloat16* q, const int32_t* sel_idx,
                           const int32_t* sel_cnt, int k_cap, __nv_bfloat16* out, float* lse, cudaStream_t s, const TailCall& tc) {
  const GroupDev& dev = grp->dev;
  const int problems = (l1 - l0) * dev.batch * dev.H_kv;
  Sched sc;
  sc.l0 = l0;
  sc.tpp = (k_cap + kTile - 1) / kTile;
  sc.n_tiles = problems * sc.tpp;
  sc.n_ctas = sc.n_tiles < grp->sm_count ? sc.n_tiles : grp->sm_count;
  sc.share = sc.n_tiles / sc.n_ctas;
  sc.extra = sc.n_tiles - sc.share * sc.n_ctas;
  sc.n_slots = fused_slots(grp);
  sc.k_cap = k_cap;
  sc.prof = grp->prof;
  static_assert(NR * WB <= 64 && WB <= kMaxBlocks, "value epilogue registers");
  const size_t smem = fused_smem_bytes<DH, NR>();
  CUtensorMap mk;
  memcpy(&mk, grp->bk_tmap, sizeof(mk));
  cudaError_t e;
  auto launch = [&](auto kernel_smem, auto kernel, int quant) {
    e = kernel_smem(smem, grp->device);
    if (e == cudaSuccess) e = launch_pdl(kernel, dim3(sc.n_ctas), dim3(fused_threads(quant)), smem, s, mk, dev, sc, q, sel_idx, sel_cnt);
  };
#define XKV_FUSED(PROF, QUANT, MMA) launch(ensure_dyn_smem<sr_fused_kernel<DH, NR, WB, PROF, QUANT, MMA>>, sr_fused_kernel<DH, NR, WB, PROF, QUANT, MMA>, QUANT)
  // up to four heads, bf16 bases, two tiles per CTA or more: packed multiply-adds (measured at quad_logits)
  const bool fma = NR == 4 && sc.n_tiles >= 2 * sc.n_ctas;
  if (grp->prof) {     // the variant with the diagnostic counters compiled in
    if (dev.Aq_k) return cudaErrorNotSupported;        // no diagnostic variant of the quantised gather
    if (fma) XKV_FUSED(true, 0, NR != 4); else XKV_FUSED(true, 0, true);
  } else if (dev.Aq_k && dev.quant_bits == 3) {
    XKV_FUSED(false, 3, true);
  } else if (dev.Aq_k) {
    XKV_FUSED(false, 4, true);
  } else if (fma) {
    XKV_FUSED(false, 0, NR != 4);
  } else {
    XKV_FUSED(false, 0, true);
  }
#undef XKV_FUSED
  if (e != cudaSuccess) return e;
  count_launch(kFamFused);
  TailParts tail{nullptr, 0};
  if (tc.k) {
    e = launch_tail_partials(grp, l0, l1, q, tc.k, tc.v, tc.len, tc.cap, tc.part, true, s);
    if (e != cudaSuccess) return e;
    tail = TailParts{tc.part, tail_splits(tc.cap)};
  }
  // one CTA per query head while those CTAs fit the SMs about twice over; beyond that one CTA per group of heads
  constexpr int HG = NR <= 4 ? 4 : 8;
  bool multi = false;
  if ((long long)problems * dev.n_rep <= 2LL * grp->sm_count) {
    const size_t msmem = sizeof(float) * (((size_t)dev.r_v + 3) / 4 * 4 + (size_t)(kMergeThreads / (DH / 8)) * DH);
    e = ensure_dyn_smem<merge_segments_kernel<DH>>(msmem, grp->device);
    if (e != cudaSuccess) return e;
    e = launch_pdl(merge_segments_kernel<DH>, dim3(problems * dev.n_rep), dim3(kMergeThreads), msmem, s, dev, sc, tail, out, lse);
  } else {
    const size_t msmem = sizeof(float) * ((size_t)HG * (((size_t)dev.r_v + 3) / 4 * 4) + (size_t)HG * (kMergeMultiThreads / 32) * DH);
    const int ngrp = (dev.n_rep + HG - 1) / HG;
    e = ensure_dyn_smem<merge_segments_multi_kernel<DH, HG>>(msmem, grp->device);
    if (e != cudaSuccess) return e;
    e = launch_pdl(merge_segments_multi_kernel<DH, HG>, dim3(problems * ngrp), dim3(kMergeMultiThreads), msmem, s, dev, sc, tail, out, lse);
    multi = true;
  }
  if (e != cudaSuccess) return e;
  count_launch(multi ? kFamMergeMulti : kFamMerge);
  return cudaGetLastError();
}

}  // namespace

// A problem never has more segments than there are CTAs + 1; the merge kernel's tables hold kMergeMaxSeg of them.
bool fused_sm_count_ok(int sm_count) { return sm_count >= 1 && sm_count + 1 <= kMergeMaxSeg; }

int fused_slots(const xkv_group* grp) {
  const int tpp_max = (grp->k_cap_max + kTile - 1) / kTile;
  return (tpp_max < grp->sm_count ? tpp_max : grp->sm_count) + 1;
}

size_t fused_part_floats(const xkv_group* grp) {
  const xkv_group_config& c = grp->cfg;
  return (size_t)c.G * c.batch * c.H_kv * fused_slots(grp) * (size_t)(c.H_q / c.H_kv) * (c.r_v + 2);
}

// The tensor-core path covers r_v up to 1024 (512 with more than 8 query heads per KV head).
bool fused_supported(const xkv_group* grp) {
  const int n_rep = grp->dev.n_rep, blocks = (grp->dev.r_v + 127) / 128;
  return blocks <= (n_rep <= 8 ? 8 : 4);
}

cudaError_t launch_fused(const xkv_group* grp, int l0, int l1, const __nv_bfloat16* q, const int32_t* sel_idx,
                         const int32_t* sel_cnt, int k_cap, __nv_bfloat16* out, float* lse, cudaStream_t s, const TailCall& tail) {
  const int n_rep = grp->dev.n_rep, blocks = (grp->dev.r_v + 127) / 128;   // WB: the smallest variant that holds r_v
#define XKV_DISPATCH(DH)                                                                                 \
  if (n_rep <= 4 && blocks <= 4) return launch_fused_t<DH, 4, 4>(grp, l0, l1, q, sel_idx, sel_cnt, k_cap, out, lse, s, tail);  \
  if (n_rep <= 4) return launch_fused_t<DH, 4, 8>(grp, l0, l1, q, sel_idx, sel_cnt, k_cap, out, lse, s, tail);  \
  if (n_rep <= 8 && blocks <= 4) return launch_fused_t<DH, 8, 4>(grp, l0, l1, q, sel_idx, sel_cnt, k_cap, out, lse, s, tail);  \
  if (n_rep <= 8) return launch_fused_t<DH, 8, 8>(grp, l0, l1, q, sel_idx, sel_cnt, k_cap, out, lse, s, tail);  \
  return launch_fused_t<DH, 16, 4>(grp, l0, l1, q, sel_idx, sel_cnt, k_cap, out, lse, s, tail);
  if (grp->dev.d_h == 128) { XKV_DISPATCH(128) }
  XKV_DISPATCH(64)
#undef XKV_DISPATCH
}

}  // namespace xkv
