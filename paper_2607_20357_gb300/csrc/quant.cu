// e4m3 operands of the gated projections (FP8 weights, which the paper
// calls orthogonal to its method, Sec. 5). Every row -- an output channel of
// a weight matrix, or an activation row feeding one of the four gated GEMMs
// -- is scaled so that its largest magnitude maps to 448, the largest finite
// e4m3 value, and rounded to nearest even with saturation:
//
//   amax = max |x|, inv = 448 / amax, scale = amax / 448 (float32, correctly
//   rounded; 0 and 0 when amax = 0), code = e4m3(x * inv).
//
// With a gain vector (the RMSNorm gain of the projection's input norm) the
// row quantised is x * gain, each product exact in float32 (two bf16
// factors). The norm's 1/rms(x) is a factor of the whole row, so the codes of
// x * gain are those of RMSNorm(x) * gain and the GEMM applies 1/rms with the
// row's scale after the product.
//
// The GEMM multiplies codes and scales its accumulator by both rows' scales.
#include <algorithm>

#include "kernels.cuh"

namespace svl {

constexpr int kQuantWarps = 8;

// Eight bf16 ones: the gain of a row quantised as it is.
SVL_DEVINL uint4 ones8() { return make_uint4(0x3F803F80u, 0x3F803F80u, 0x3F803F80u, 0x3F803F80u); }

// The eight values of a 16-byte chunk times their gains, in float32 (exact:
// the product of two bf16 values has at most 16 significant bits).
SVL_DEVINL void scaled8(const uint4 x, const uint4 g, float f[8]) {
  const uint32_t xw[4] = {x.x, x.y, x.z, x.w}, gw[4] = {g.x, g.y, g.z, g.w};
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const float2 a = unpack_bf16x2(xw[q]), b = unpack_bf16x2(gw[q]);
    f[2 * q] = __fmul_rn(a.x, b.x);
    f[2 * q + 1] = __fmul_rn(a.y, b.y);
  }
}

// What is computed from x before is computed again after this.
SVL_DEVINL void opaque(uint4& x) { asm volatile("" : "+r"(x.x), "+r"(x.y), "+r"(x.z), "+r"(x.w)); }

// e4m3 codes of eight values times inv (each product rounded to float32).
SVL_DEVINL uint2 codes8(const float f[8], float inv) {
  uint2 o;
  o.x = static_cast<uint32_t>(e4m3x2(__fmul_rn(f[0], inv), __fmul_rn(f[1], inv))) |
        (static_cast<uint32_t>(e4m3x2(__fmul_rn(f[2], inv), __fmul_rn(f[3], inv))) << 16);
  o.y = static_cast<uint32_t>(e4m3x2(__fmul_rn(f[4], inv), __fmul_rn(f[5], inv))) |
        (static_cast<uint32_t>(e4m3x2(__fmul_rn(f[6], inv), __fmul_rn(f[7], inv))) << 16);
  return o;
}

// The same two in packed arithmetic, two values in a 64-bit register: the eight
// values of a chunk (times their gains), their largest magnitude with m, and
// their codes. (The row kernel is bound by issue slots as much as by memory.)
SVL_DEVINL uint64_t mul2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
SVL_DEVINL uint64_t bf16_pair(uint32_t w) {
  return (static_cast<uint64_t>(w & 0xFFFF0000u) << 32) | (w << 16);
}
SVL_DEVINL float pair_lo(uint64_t v) { return __uint_as_float(static_cast<uint32_t>(v)); }
SVL_DEVINL float pair_hi(uint64_t v) { return __uint_as_float(static_cast<uint32_t>(v >> 32)); }

template <bool GAIN>
SVL_DEVINL void products8(const uint4& x, const uint4& g, uint64_t f[4]) {
  const uint32_t xw[4] = {x.x, x.y, x.z, x.w}, gw[4] = {g.x, g.y, g.z, g.w};
#pragma unroll
  for (int q = 0; q < 4; ++q) f[q] = GAIN ? mul2(bf16_pair(xw[q]), bf16_pair(gw[q])) : bf16_pair(xw[q]);
}

SVL_DEVINL float max_abs8(const uint64_t f[4], float m) {
#pragma unroll
  for (int q = 0; q < 4; ++q)
    asm("max.f32 %0, %1, %2, %3;" : "=f"(m) : "f"(m), "f"(fabsf(pair_lo(f[q]))), "f"(fabsf(pair_hi(f[q]))));
  return m;
}

SVL_DEVINL uint2 codes8(const uint64_t f[4], uint64_t inv2) {
  uint32_t c[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const uint64_t v = mul2(f[q], inv2);
    c[q] = e4m3x2(pair_lo(v), pair_hi(v));
  }
  return make_uint2(c[0] | (c[1] << 16), c[2] | (c[3] << 16));
}

// One warp per row, two passes (rows wider than 16,384 codes).
__global__ void __launch_bounds__(kQuantWarps * 32) quant_rows_kernel(QuantArgs a) {
  pdl_begin(a.late);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t r = static_cast<int64_t>(blockIdx.x) * kQuantWarps + warp;
  int64_t rows = a.rows;
  if (a.cu_seqlens) rows = min(rows, static_cast<int64_t>(a.cu_seqlens[a.B]));
  if (r >= rows) return;
  int mask = (1 << a.G) - 1;
  if (a.group_gate && a.l >= a.P) {
    const int b = find_sample(a.cu_seqlens, a.B, static_cast<int>(r));
    const size_t bl = static_cast<size_t>(b) * a.L + a.l;
    mask = 0;
    if (a.layer_gate[bl])
      for (int j = 0; j < a.G; ++j) mask |= a.group_gate[bl * a.G + j] ? (1 << j) : 0;
  }
  const __nv_bfloat16* src = a.src + r * a.ld_src;
  float amax = 0.f;
  for (int j = 0; j < a.G; ++j) {
    if (!((mask >> j) & 1)) continue;
    const uint4* s4 = reinterpret_cast<const uint4*>(src + static_cast<size_t>(j) * a.kg);
    const uint4* g4 = a.gain ? reinterpret_cast<const uint4*>(a.gain + static_cast<size_t>(j) * a.kg) : nullptr;
    for (int c = lane; c < a.kg / 8; c += 32) {
      float f[8];
      scaled8(s4[c], g4 ? g4[c] : ones8(), f);
#pragma unroll
      for (int q = 0; q < 8; ++q) amax = fmaxf(amax, fabsf(f[q]));
    }
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, off));
  const float inv = amax > 0.f ? __fdiv_rn(448.f, amax) : 0.f;
  uint8_t* dst = a.dst + r * a.ld_dst;
  for (int j = 0; j < a.G; ++j) {
    const bool on = (mask >> j) & 1;
    const uint4* s4 = reinterpret_cast<const uint4*>(src + static_cast<size_t>(j) * a.kg);
    const uint4* g4 = a.gain ? reinterpret_cast<const uint4*>(a.gain + static_cast<size_t>(j) * a.kg) : nullptr;
    uint2* d8 = reinterpret_cast<uint2*>(dst + static_cast<size_t>(j) * a.kgp);
    for (int c = lane; c < a.kgp / 8; c += 32) {
      uint2 o = make_uint2(0, 0);
      if (on && c < a.kg / 8) {
        float f[8];
        scaled8(s4[c], g4 ? g4[c] : ones8(), f);
        o = codes8(f, inv);
      }
      d8[c] = o;
    }
  }
  if (lane == 0) a.scale[r] = amax > 0.f ? __fdiv_rn(amax, 448.f) : 0.f;
}

// 128-thread CTAs walking the rows (row = blockIdx.x + i * gridDim.x, so a
// grid of the CTAs that fit serves any row count): thread t holds the row's
// 16-byte chunks t, t + 128, ... (NCH of them) in registers between the amax
// and the code pass, so each bf16 value is read once. Bound by memory (2 bytes
// in, 1 out per value), so nothing but the row's own load and reduction may lie
// on a row's chain: the group masks of the CTA's next 128 rows are looked up
// together, a row per thread (the search of the sample and its gates are six
// dependent loads), the gain's chunks are read once, and the next row loads
// while this one is reduced. 5,400 rows, 11,008 wide: 45 -> 30 us (0.88 of the
// measured copy bandwidth); 4,096 wide with gains: 19 -> 16 us (a few rows per
// CTA, so the launch and the first loads weigh more).
constexpr int kQuantThreads = 128;
constexpr int kColMask = (1 << 26) - 1;

template <int NCH, bool GAIN>
__global__ void __launch_bounds__(kQuantThreads, NCH <= 4 ? 7 : NCH <= 12 ? 4 : 3) quant_row_cta_kernel(QuantArgs a) {
  __shared__ float red[2][kQuantThreads / 32];
  __shared__ int s_mask[kQuantThreads];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int per_g = a.kgp / 8, src_per_g = a.kg / 8, nchunk = a.G * per_g;
  const bool gated = a.group_gate && a.l >= a.P;
  int col[NCH];  // source column of each chunk, its group in the top bits; group 31: padding (never in a mask)
  uint4 gv[GAIN ? NCH : 1];
#pragma unroll
  for (int i = 0; i < NCH; ++i) {
    const int c = tid + i * kQuantThreads, j = c / per_g, cc = c - j * per_g;
    const bool src = c < nchunk && cc < src_per_g;
    col[i] = src ? (j << 26) | (j * a.kg + cc * 8) : static_cast<int>(31u << 26);
  }
  pdl_begin(a.late);
  // (the gain too may come from the launch before: svl_quantize_rows_e4m3 takes a caller's vector)
  if constexpr (GAIN) {
#pragma unroll
    for (int i = 0; i < NCH; ++i)
      gv[i] = static_cast<unsigned>(col[i]) >> 26 != 31u ? *reinterpret_cast<const uint4*>(a.gain + (col[i] & kColMask))
                                                         : ones8();
  }
  int64_t rows = a.rows;
  if (a.cu_seqlens) rows = min(rows, static_cast<int64_t>(a.cu_seqlens[a.B]));
  auto load = [&](int64_t r, int mask, uint4* v) {
    const __nv_bfloat16* src = a.src + r * a.ld_src;
#pragma unroll
    for (int i = 0; i < NCH; ++i) {
      v[i] = make_uint4(0, 0, 0, 0);
      if ((mask >> (static_cast<unsigned>(col[i]) >> 26)) & 1)
        v[i] = *reinterpret_cast<const uint4*>(src + (col[i] & kColMask));
    }
  };
  const int all = (1 << a.G) - 1;
  uint4 v[NCH];
  int n = 0;  // rows done
  for (int64_t r = blockIdx.x; r < rows; r += gridDim.x, ++n) {
    const int64_t next = r + gridDim.x;
    if (gated && n % kQuantThreads == 0) {
      if (n > 0) __syncthreads();  // the masks of the rows before have been read
      const int64_t rm = r + static_cast<int64_t>(tid) * gridDim.x;
      int mask = 0;
      if (rm < rows) {
        const int b = find_sample(a.cu_seqlens, a.B, static_cast<int>(rm));
        const size_t bl = static_cast<size_t>(b) * a.L + a.l;
        if (a.layer_gate[bl])
          for (int j = 0; j < a.G; ++j) mask |= a.group_gate[bl * a.G + j] ? (1 << j) : 0;
      }
      s_mask[tid] = mask;
      __syncthreads();
    }
    if (n % kQuantThreads == 0) load(r, gated ? s_mask[0] : all, v);
    float amax = 0.f;
#pragma unroll
    for (int i = 0; i < NCH; ++i) {
      uint64_t f[4];
      if (GAIN) opaque(gv[i]);
      products8<GAIN>(v[i], gv[GAIN ? i : 0], f);
      amax = max_abs8(f, amax);
    }
    uint4 vn[NCH];  // (the first row of a batch of masks is loaded above)
    if (next < rows && (n + 1) % kQuantThreads != 0) load(next, gated ? s_mask[(n + 1) % kQuantThreads] : all, vn);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, off));
    float* rd = red[n & 1];  // the slots alternate between consecutive rows
    if (lane == 0) rd[warp] = amax;
    __syncthreads();
    amax = fmaxf(fmaxf(rd[0], rd[1]), fmaxf(rd[2], rd[3]));
    const float inv = amax > 0.f ? __fdiv_rn(448.f, amax) : 0.f;
    const uint64_t inv2 = (static_cast<uint64_t>(__float_as_uint(inv)) << 32) | __float_as_uint(inv);
    uint8_t* dst = a.dst + r * a.ld_dst;
#pragma unroll
    for (int i = 0; i < NCH; ++i) {
      const int c = tid + i * kQuantThreads;
      if (c < nchunk) {
        // (converted again: 8 values a chunk kept since the first pass would take
        // the registers of four more resident CTAs)
        opaque(v[i]);
        if (GAIN) opaque(gv[i]);
        uint64_t f[4];
        products8<GAIN>(v[i], gv[GAIN ? i : 0], f);
        // chunk c of the padded row sits at byte 8 c (groups are kgp apart)
        *reinterpret_cast<uint2*>(dst + static_cast<size_t>(c) * 8) = codes8(f, inv2);
      }
      v[i] = vn[i];
    }
    if (tid == 0) a.scale[r] = amax > 0.f ? __fdiv_rn(amax, 448.f) : 0.f;
  }
}

// A grid of the CTAs that fit on the device at once.
template <int NCH, bool GAIN>
static cudaError_t launch_row_cta(const QuantArgs& a, cudaStream_t s) {
  static int resident = 0;
  if (!resident) {
    int dev = 0, sms = 0, per_sm = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess)
      e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, quant_row_cta_kernel<NCH, GAIN>, kQuantThreads, 0);
    if (e != cudaSuccess) return e;
    resident = std::max(sms * per_sm, 1);
  }
  const dim3 grid(static_cast<unsigned>(std::min<int64_t>(a.rows, resident)));
  return launch_pdl(quant_row_cta_kernel<NCH, GAIN>, grid, kQuantThreads, 0, s, a);
}

cudaError_t launch_quant_rows(const QuantArgs& a, cudaStream_t s) {
  if (a.rows <= 0) return cudaSuccess;
  const int64_t chunks = static_cast<int64_t>(a.G) * (a.kgp / 8);
  if (a.gain) {
    // gain rows (QKV and gate/up inputs): the gain chunks stay in registers too
    if (chunks <= 4 * kQuantThreads) return launch_row_cta<4, true>(a, s);
    if (chunks <= 8 * kQuantThreads) return launch_row_cta<8, true>(a, s);
  } else {
    if (chunks <= 4 * kQuantThreads) return launch_row_cta<4, false>(a, s);
    if (chunks <= 8 * kQuantThreads) return launch_row_cta<8, false>(a, s);
    if (chunks <= 12 * kQuantThreads) return launch_row_cta<12, false>(a, s);
    if (chunks <= 16 * kQuantThreads) return launch_row_cta<16, false>(a, s);
  }
  const int64_t blocks = (a.rows + kQuantWarps - 1) / kQuantWarps;
  return launch_pdl(quant_rows_kernel, dim3(static_cast<unsigned>(blocks)), kQuantWarps * 32, 0, s, a);
}

}  // namespace svl
