// Round-to-nearest quantisation of the factorised cache (App. "Integrate with Quantization": "a simple
// round-to-nearest (RTN) quantization method to the compressed cache"; 4 bits give 8.03x -> 25.7x, i.e. 5 stored
// bits per scalar).  Groups of 32 consecutive scalars of a row share a bf16 scale and a bf16 offset:
//   zero = bf16(min), scale = bf16((max - min) / 15), code = clip(rint((x - zero) / scale), 0, 15)   (fp32, IEEE)
//   x_hat = bf16(code * scale + zero)                                   (one rounding of the exact value)
// (4 bits; the 3-bit variant divides by 7, clips at 7 and stores 16-byte records, see dequant_group3.)
// Storage: codes, 4 bits each, [rows][cols/2] bytes; inside every 32-bit word (8 consecutive scalars e0..e7) the
// low half holds e0, e2, e4, e6 and the high half e1, e3, e5, e7 (nibble k of each half), so that
// (word >> 4k) & 0x000F000F is the pair (e_2k, e_2k+1) in the two halves of a register -- the form the packed
// bf16 arithmetic of the gather wants.  meta, [rows][cols/32] 32-bit words: scale in the low half, offset in the high.
#include "xkv_internal.cuh"
#include "xkv_ptx.cuh"

namespace xkv {

namespace {

constexpr int kQuantThreads = 256;
// The first blocks, those that may start while the kernel before still runs, have their scalars brought into L2 before
// they wait for it (the second level is where that kernel's writes would land, so nothing stale is read): six launches of a
// window 41.9 -> 40.6 us.  As many as an SM's 2048 threads hold of them; its registers hold five at a time, but the others
// follow before those have finished (five per SM: 41.2 us).  A device with another number of SMs only prefetches more or less.
constexpr int kQuantAhead = 2048 / kQuantThreads * kPlanSms;
constexpr int kQuantPieces = 4;    // 16-byte pieces per thread, all requested before the first is used (four: see the quantiser)

__device__ __forceinline__ uint32_t min_bf16x2(uint32_t a, uint32_t b) {
  uint32_t r;
  asm("min.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
  return r;
}
__device__ __forceinline__ uint32_t max_bf16x2(uint32_t a, uint32_t b) {
  uint32_t r;
  asm("max.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
  return r;
}
// ... and with a NaN as the result where one of the two is
__device__ __forceinline__ uint32_t max_nan_bf16x2(uint32_t a, uint32_t b) {
  uint32_t r;
  asm("max.NaN.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
  return r;
}
__device__ __forceinline__ float max_nan(float a, float b) {
  float r;
  asm("max.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
  return r;
}

// HBM bound: 2 bytes read and (bits + 1) / 8 written per scalar.  Four consecutive lanes share a group of 32 scalars, a
// lane holds one 16-byte piece (8 scalars) of four groups: loads and stores of a warp are contiguous, extrema are packed
// bf16 minima and maxima, folded by halving so that a lane ends with those of one group.
// The codes are rint(fl(f / scale)), f = x - zero.  The correctly rounded quotient comes from the correctly rounded
// reciprocal y by q = f y, q + (f - q scale) y with fused multiply-adds (Markstein, IBM J. Res. Dev. 34(1), 1990); the
// exact quotient of a 24-bit by an 8-bit number is never closer than 2^-33 to a rounding boundary and the value that is
// rounded last is off by less than 2^-46, so every bit is that of the division.  Half-integers are common here
// (differences of bf16 numbers over a bf16 scale): the quotient has to be exact, a test with a fallback diverged in most
// warps (25 us for 65536 x 384 scalars, with an IEEE division per scalar and one thread per group 38 us; this form 19.5, and 17 with
// two scalars per packed instruction).
// A group's scale, offset and reciprocal are some forty instructions, a quarter of the kernel's when all four lanes worked
// them out for every group, and instruction issue is what bounds it (71 % of the slots now): a quad holds four groups, and lane p
// does that work for group p alone.  A window's token bases and matrices (65536 rows of 384 and 576; six launches):
// 46.4 -> 41.8 us.
// Rounding goes through 1.5 * 2^23, whose sum with the quotient holds the integer in its low bits.
constexpr float kRintMagic = 12582912.0f;

template <int BITS>
__device__ __forceinline__ uint32_t rtn_code_exact(float f, float scale) {
  constexpr float kTop = (float)((1 << BITS) - 1);
  float q = 0.0f;
  if (scale > 0.0f) q = rintf(__fdiv_rn(f, scale));          // ties to even
  return (uint32_t)fminf(fmaxf(q, 0.0f), kTop);
}

template <int BITS>
__global__ void __launch_bounds__(kQuantThreads)
quantize_rtn_kernel(const uint4* __restrict__ x, long long n_pieces, uint32_t* __restrict__ codes, uint32_t* __restrict__ meta) {
  static_assert(kQuantPieces == 4, "a group for every lane of a quad");
  constexpr float kTop = (float)((1 << BITS) - 1);
  const int p = threadIdx.x & 3;                           // piece of the group; n_pieces is a multiple of 4
  const long long first = (long long)blockIdx.x * (kQuantThreads * kQuantPieces) + threadIdx.x;
  if (blockIdx.x < kQuantAhead && (threadIdx.x & 7) == 0) {
#pragma unroll
    for (int u = 0; u < kQuantPieces; ++u)
      if (first + u * kQuantThreads < n_pieces) asm volatile("prefetch.global.L2 [%0];" ::"l"(x + first + u * kQuantThreads));
  }
  ptx::grid_dependency_wait();
  ptx::grid_dependency_launch();
  uint4 v[kQuantPieces];
#pragma unroll
  for (int u = 0; u < kQuantPieces; ++u) {
    const long long i = first + u * kQuantThreads;
    v[u] = i < n_pieces ? __ldcs(x + i) : make_uint4(0u, 0u, 0u, 0u);
  }
  // The extrema of the quad's four groups, folded by halving: lane p ends with those of its group first + p * kQuantThreads,
  // works out scale, offset and reciprocal of that group alone, and the quad passes them round.
  uint32_t lo2[kQuantPieces], hi2[kQuantPieces];
#pragma unroll
  for (int u = 0; u < kQuantPieces; ++u) {
    lo2[u] = min_bf16x2(min_bf16x2(v[u].x, v[u].y), min_bf16x2(v[u].z, v[u].w));
    hi2[u] = max_nan_bf16x2(max_nan_bf16x2(v[u].x, v[u].y), max_nan_bf16x2(v[u].z, v[u].w));
  }
#pragma unroll
  for (int o = 1; o < kQuantPieces; o <<= 1) {
    const bool up = (p & o) != 0;
#pragma unroll
    for (int i = 0; i + o < kQuantPieces; i += 2 * o) {
      const uint32_t lo_up = __shfl_xor_sync(0xffffffffu, up ? lo2[i] : lo2[i + o], o);
      const uint32_t hi_up = __shfl_xor_sync(0xffffffffu, up ? hi2[i] : hi2[i + o], o);
      lo2[i] = min_bf16x2(up ? lo2[i + o] : lo2[i], lo_up);
      hi2[i] = max_nan_bf16x2(up ? hi2[i + o] : hi2[i], hi_up);
    }
  }
  uint32_t own_meta;
  float own_y;                                             // reciprocal of the scale, 0: see below
  {
    const float lo = fminf(__uint_as_float(lo2[0] << 16), __uint_as_float(lo2[0] & 0xffff0000u));
    const float hi = max_nan(__uint_as_float(hi2[0] << 16), __uint_as_float(hi2[0] & 0xffff0000u));
    const __nv_bfloat16 zb = __float2bfloat16_rn(lo);
    const __nv_bfloat16 sb = __float2bfloat16_rn(__fdiv_rn(__fsub_rn(hi, lo), kTop));
    const float scale = __bfloat162float(sb);
    own_y = scale >= 1e-30f && scale <= 1e30f ? __frcp_rn(scale) : 0.0f;
    own_meta = (uint32_t)__bfloat16_as_ushort(sb) | ((uint32_t)__bfloat16_as_ushort(zb) << 16);
  }
#pragma unroll
  for (int u = 0; u < kQuantPieces; ++u) {
    const uint32_t w[4] = {v[u].x, v[u].y, v[u].z, v[u].w};
    uint32_t mw = __shfl_sync(0xffffffffu, own_meta, u, 4);
    const float y = __shfl_sync(0xffffffffu, own_y, u, 4);
    const float scale = __uint_as_float(mw << 16), zero = __uint_as_float(mw & 0xffff0000u);
    // two scalars per packed instruction; m: rint(quotient) + kRintMagic of the pairs (2e, 2e + 1)
    ptx::u64 f[4], m[4];
    const ptx::u64 nz2 = ptx::pack2(-zero, -zero);
#pragma unroll
    for (int e = 0; e < 4; ++e) f[e] = ptx::add2(ptx::pack2(__uint_as_float(w[e] << 16), __uint_as_float(w[e] & 0xffff0000u)), nz2);
    // constant groups, scales with an imprecise or overflowing reciprocal, infinities: the division for every scalar.  A NaN
    // (code 0, no part in the extrema) leads here by way of the maximum, so that it costs the other groups nothing (a
    // clamp of every code took 65536 x 960 scalars from 46.1 to 48.1 us); the maximum is taken again without it.
    if (y == 0.0f) {
      float step = scale;
      if (isnan(scale)) {
        const unsigned quad = 0xfu << (threadIdx.x & 28u);  // (the same branch in the four lanes of a group)
        uint32_t top2 = max_bf16x2(max_bf16x2(w[0], w[1]), max_bf16x2(w[2], w[3]));
#pragma unroll
        for (int o = 1; o < 4; o <<= 1) top2 = max_bf16x2(top2, __shfl_xor_sync(quad, top2, o));
        const float top = fmaxf(__uint_as_float(top2 << 16), __uint_as_float(top2 & 0xffff0000u));
        const __nv_bfloat16 sb = __float2bfloat16_rn(__fdiv_rn(__fsub_rn(top, zero), kTop));
        step = __bfloat162float(sb);
        mw = (mw & 0xffff0000u) | (uint32_t)__bfloat16_as_ushort(sb);
        if (p == u) own_meta = mw;
      }
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const float2 x2 = ptx::unpack2(f[e]);
        m[e] = ptx::pack2((float)rtn_code_exact<BITS>(x2.x, step) + kRintMagic, (float)rtn_code_exact<BITS>(x2.y, step) + kRintMagic);
      }
    } else {
      const ptx::u64 y2 = ptx::pack2(y, y), ns2 = ptx::pack2(-scale, -scale), magic2 = ptx::pack2(kRintMagic, kRintMagic);
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const ptx::u64 t = ptx::mul2(f[e], y2);
        m[e] = ptx::add2(ptx::fma2(ptx::fma2(t, ns2, f[e]), y2, t), magic2);
      }
    }
    // A pair of codes as the low and the high half of a word: f is at least 0 and at most kTop * scale * (1 + 2^-8), so the
    // sixteen low bits of m are the code.
    uint32_t c[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const float2 x2 = ptx::unpack2(m[e]);
      c[e] = __byte_perm(__float_as_uint(x2.x), __float_as_uint(x2.y), 0x5410);
    }
    uint32_t word = 0;
    if constexpr (BITS == 4) {
      word = (((c[3] << 4) + c[2]) << 8) + ((c[1] << 4) + c[0]);
    } else {
      // the quad's 32 codes as four words of nibbles; lane 0 keeps the scale/offset word, lane j + 1 builds w_j
#pragma unroll
      for (int e = 0; e < 4; ++e) word |= ((c[e] & 0xffffu) | (c[e] >> 12)) << (8 * e);
      uint32_t n[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) n[i] = __shfl_sync(0xffffffffu, word, i, 4);
      const uint32_t a = p == 1 ? n[0] : p == 2 ? __funnelshift_r(n[1], n[2], 8) : __funnelshift_r(n[2], n[3], 16);
      const uint32_t b = p == 1 ? n[1] : p == 2 ? n[2] >> 8 : n[3] >> 16;
      word = 0;
#pragma unroll
      for (int k = 0; k < 4; ++k) word |= ((a >> (8 * k)) & 7u) << (3 * k) | ((a >> (8 * k + 4)) & 7u) << (3 * k + 16);
      word |= (b & 7u) << 12 | ((b >> 4) & 7u) << 28;
      word |= ((n[3] >> (24 + p - 1)) & 1u) << 15 | ((n[3] >> (28 + p - 1)) & 1u) << 31;
      if (p == 0) word = mw;
    }
    const long long i = first + u * kQuantThreads;
    if (i < n_pieces) {
      __stcs(codes + i, word);
    }
  }
  const long long own = first + p * kQuantThreads;         // a piece of this lane's group
  if (BITS == 4 && own < n_pieces) __stcs(meta + (own >> 2), own_meta);
}

// x_hat: bf16(code * scale + zero) with a single rounding (the packed bf16 fused multiply-add rounds the exact value
// once; small integers are exact in bf16).  One thread per 8 scalars, so that the 16-byte stores of a warp are contiguous.
__global__ void __launch_bounds__(kQuantThreads)
dequantize_rtn4_kernel(const uint32_t* __restrict__ codes, const uint32_t* __restrict__ meta, long long n_pieces,
                       uint4* __restrict__ x) {
  const long long first = (long long)blockIdx.x * (kQuantThreads * kQuantPieces) + threadIdx.x;
  ptx::grid_dependency_wait();
  ptx::grid_dependency_launch();
  uint32_t w[kQuantPieces], m[kQuantPieces];
#pragma unroll
  for (int u = 0; u < kQuantPieces; ++u) {
    const long long i = first + u * kQuantThreads;
    w[u] = i < n_pieces ? __ldg(codes + i) : 0u;
    m[u] = i < n_pieces ? __ldg(meta + (i >> 2)) : 0u;
  }
#pragma unroll
  for (int u = 0; u < kQuantPieces; ++u) {
    const long long i = first + u * kQuantThreads;
    uint32_t o[4];
    ptx::dequant_word(w[u], m[u], o);
    if (i < n_pieces) x[i] = make_uint4(o[0], o[1], o[2], o[3]);
  }
}

// The 3-bit variant, one thread per 16-byte record; the 64 bytes of a group go through shared memory so that the
// stores of a warp are contiguous (unit u of group g sits at g * 4 + (u ^ (g / 2 % 4)): no bank conflicts either way).
__global__ void __launch_bounds__(kQuantThreads)
dequantize_rtn3_kernel(const uint4* __restrict__ rec, long long n_groups, uint4* __restrict__ x) {
  __shared__ uint4 stage[kQuantThreads * 4];
  const int tid = threadIdx.x;
  const long long g0 = (long long)blockIdx.x * kQuantThreads;
  ptx::grid_dependency_wait();
  ptx::grid_dependency_launch();
  if (g0 + tid < n_groups) {
    const uint4 r = rec[g0 + tid];
    uint32_t o[16];
    ptx::dequant_group3(r.x, r.y, r.z, r.w, o);
#pragma unroll
    for (int i = 0; i < 4; ++i) stage[tid * 4 + (i ^ ((tid >> 1) & 3))] = make_uint4(o[4 * i], o[4 * i + 1], o[4 * i + 2], o[4 * i + 3]);
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int e = tid + i * kQuantThreads, g = e >> 2;
    if (g0 + g < n_groups) x[g0 * 4 + e] = stage[g * 4 + ((e & 3) ^ ((g >> 1) & 3))];
  }
}

// Blocks for n items, `per` to a block; false if there are too many for a grid.
bool blocks_for(long long n, int per, unsigned* blocks) {
  const long long b = (n + per - 1) / per;
  *blocks = (unsigned)b;
  return b <= 0x7fffffffLL;
}

}  // namespace

cudaError_t launch_quantize_rtn3(const __nv_bfloat16* x, long long rows, int cols, void* rec, cudaStream_t s) {
  const long long n_pieces = rows * (cols / 8);
  if (n_pieces == 0) return cudaSuccess;
  unsigned blocks;
  if (!blocks_for(n_pieces, kQuantThreads * kQuantPieces, &blocks)) return cudaErrorInvalidValue;
  count_launch(kFamPrep);
  return launch_pdl(quantize_rtn_kernel<3>, dim3(blocks), dim3(kQuantThreads), 0, s, (const uint4*)x, n_pieces, (uint32_t*)rec,
                    (uint32_t*)nullptr);
}

cudaError_t launch_dequantize_rtn3(const void* rec, long long rows, int cols, __nv_bfloat16* x, cudaStream_t s) {
  const long long n_groups = rows * (cols / 32);
  if (n_groups == 0) return cudaSuccess;
  unsigned blocks;
  if (!blocks_for(n_groups, kQuantThreads, &blocks)) return cudaErrorInvalidValue;
  count_launch(kFamPrep);
  return launch_pdl(dequantize_rtn3_kernel, dim3(blocks), dim3(kQuantThreads), 0, s, (const uint4*)rec, n_groups, (uint4*)x);
}

cudaError_t launch_quantize_rtn4(const __nv_bfloat16* x, long long rows, int cols, void* codes, void* meta, cudaStream_t s) {
  const long long n_pieces = rows * (cols / 8);
  if (n_pieces == 0) return cudaSuccess;
  unsigned blocks;
  if (!blocks_for(n_pieces, kQuantThreads * kQuantPieces, &blocks)) return cudaErrorInvalidValue;
  count_launch(kFamPrep);
  return launch_pdl(quantize_rtn_kernel<4>, dim3(blocks), dim3(kQuantThreads), 0, s, (const uint4*)x, n_pieces, (uint32_t*)codes,
                    (uint32_t*)meta);
}

cudaError_t launch_dequantize_rtn4(const void* codes, const void* meta, long long rows, int cols, __nv_bfloat16* x,
                                   cudaStream_t s) {
  const long long n_pieces = rows * (cols / 8);
  if (n_pieces == 0) return cudaSuccess;
  unsigned blocks;
  if (!blocks_for(n_pieces, kQuantThreads * kQuantPieces, &blocks)) return cudaErrorInvalidValue;
  count_launch(kFamPrep);
  return launch_pdl(dequantize_rtn4_kernel, dim3(blocks), dim3(kQuantThreads), 0, s, (const uint32_t*)codes, (const uint32_t*)meta,
                    n_pieces, (uint4*)x);
}

}  // namespace xkv
