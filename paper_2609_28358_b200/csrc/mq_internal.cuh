// Internal declarations shared by the library's translation units (not part of the ABI).
#pragma once

#include <cuda_runtime.h>
#include <cuda_fp16.h>
#include <cuda_fp8.h>
#include <cuda_fp4.h>
#include <cuda_fp6.h>
#include <stdint.h>

#include <atomic>

#include "mq.h"

namespace mq {

// Derived geometry of one layer (Sec. II-A) and of its stored tensors (Sec. IV-A/B).
struct Geom {
  int N, Cin, H, W, Cout, Kh, Kw, sh, sw, ph, pw;
  int Ho, Wo;
  int Cp, Cop;  // channels rounded up to 32
  int Nt;       // ceil(N / 32)
  int Ct, Cot;  // Cp / 32, Cop / 32
};

inline Geom make_geom(const mq_conv_desc& d) {
  Geom g;
  g.N = d.N; g.Cin = d.C_in; g.H = d.H; g.W = d.W; g.Cout = d.C_out; g.Kh = d.Kh; g.Kw = d.Kw;
  g.sh = d.stride_h; g.sw = d.stride_w; g.ph = d.pad_h; g.pw = d.pad_w;
  g.Ho = (d.H + 2 * d.pad_h - d.Kh) / d.stride_h + 1;
  g.Wo = (d.W + 2 * d.pad_w - d.Kw) / d.stride_w + 1;
  g.Cp = (d.C_in + 31) / 32 * 32;
  g.Cop = (d.C_out + 31) / 32 * 32;
  g.Nt = (d.N + 31) / 32;
  g.Ct = g.Cp / 32;
  g.Cot = g.Cop / 32;
  return g;
}

__host__ __device__ inline int fmt_bits(int fmt) { return fmt == MQ_E2M1 ? 4 : 8; }
__host__ __device__ inline int fmt_emax(int fmt) { return fmt == MQ_E4M3 ? 8 : (fmt == MQ_E5M2 ? 15 : (fmt == MQ_E3M2 ? 4 : 2)); }
__host__ __device__ inline bool fmt_is_6bit(int fmt) { return fmt == MQ_E3M2 || fmt == MQ_E2M3; }
// packed 6-bit storage: the same element formats, 16 codes in 12 bytes
__host__ __device__ inline bool fmt_is_packed6(int fmt) { return fmt == MQ_E3M2_P6 || fmt == MQ_E2M3_P6; }
__host__ __device__ inline int fmt_base(int fmt) { return fmt == MQ_E3M2_P6 ? MQ_E3M2 : (fmt == MQ_E2M3_P6 ? MQ_E2M3 : fmt); }
__host__ __device__ inline int fmt_store_bits(int fmt) { return fmt_is_packed6(fmt) ? 6 : fmt_bits(fmt); }
// 16 one-byte 6-bit codes (four words) -> the 96-bit field of the packed storage: code k in bits 6k .. 6k+5
__host__ __device__ inline void pack6x16(const uint32_t w[4], uint32_t out[3]) {
  uint32_t t[4];
  for (int i = 0; i < 4; ++i) t[i] = (w[i] & 0x3Fu) | ((w[i] >> 2) & 0xFC0u) | ((w[i] >> 4) & 0x3F000u) | ((w[i] >> 6) & 0xFC0000u);
  out[0] = t[0] | (t[1] << 24);
  out[1] = (t[1] >> 8) | (t[2] << 16);
  out[2] = (t[2] >> 16) | (t[3] << 8);
}
// and back: the field's three words -> 16 one-byte codes
__host__ __device__ inline void unpack6x16(const uint32_t in[3], uint32_t w[4]) {
  uint32_t t[4];
  t[0] = in[0] & 0xFFFFFFu;
  t[1] = ((in[0] >> 24) | (in[1] << 8)) & 0xFFFFFFu;
  t[2] = ((in[1] >> 16) | (in[2] << 16)) & 0xFFFFFFu;
  t[3] = in[2] >> 8;
  for (int i = 0; i < 4; ++i) w[i] = (t[i] & 0x3Fu) | ((t[i] & 0xFC0u) << 2) | ((t[i] & 0x3F000u) << 4) | ((t[i] & 0xFC0000u) << 6);
}
// format field of the tcgen05 instruction descriptor (kind::mxf8f6f4)
__host__ __device__ inline unsigned fmt_mma_code(int fmt) { return fmt == MQ_E4M3 ? 0u : (fmt == MQ_E5M2 ? 1u : (fmt == MQ_E2M3 ? 3u : (fmt == MQ_E3M2 ? 4u : 5u))); }

// Number of kernels the library has launched in this process (diagnostic; see mq_kernel_launch_count).
void count_launches(int n);

// Streaming multiprocessors of the current device (148 on a B200); grids are sized in multiples of it.
inline int sm_count() {
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms <= 0) return 148;
  return sms;
}

// Integer value of an MQ_* environment knob.  Each knob is read from the environment ONCE, on its first use in the
// process, and answered from a table afterwards, so that a size query and the call it sizes always see the same plan;
// mq_reload_env() (a diagnostic entry point) empties the table.
// A call asks for some dozens of knobs, so every place that asks keeps the table's answer beside it, stamped with the
// table's generation: one atomic load instead of a lock, a string and a map (the latter were 1-2 us of each call).
extern std::atomic<uint32_t> g_env_generation;   // 31 bits, advanced by mq_reload_env
uint64_t env_lookup(const char* name);           // generation << 33 | set << 32 | value, from the table
class EnvKnob {
 public:
  constexpr explicit EnvKnob(const char* name) : name_(name) {}
  int get(int dflt) {
    uint64_t c = cell_.load(std::memory_order_acquire);
    if ((uint32_t)(c >> 33) != (g_env_generation.load(std::memory_order_acquire) & 0x7fffffffu)) {
      c = env_lookup(name_);
      cell_.store(c, std::memory_order_release);
    }
    return (c >> 32) & 1u ? (int)(uint32_t)c : dflt;
  }

 private:
  const char* name_;
  std::atomic<uint64_t> cell_{0};
};
#define MQ_ENV(name, dflt) ([]() -> ::mq::EnvKnob& { static ::mq::EnvKnob knob(name); return knob; }().get(dflt))

// ---- launchers (defined in the .cu files) ---------------------------------------------------
struct QuantArgs {
  const float* src;
  uint8_t* codes;
  uint8_t* scales;
  int P, R, C, Cp;                 // positions, rows of the 2-D view, channels, padded channels
  long long out_stride_p, out_stride_r;  // in elements of the codes tensor
  long long sc_stride_p, sc_stride_r;    // in scale bytes
  int fmt;
  // source strides in floats when the source has the channel axis fastest (fp32 [H][W][N][C] / [Cout][Kh][Kw][Cin]):
  // element (p, r, c) at p * src_stride_p + r * src_stride_r + c; both zero for the NCHW / OIHW source
  long long src_stride_p, src_stride_r;
  // stochastic rounding (Eq. 6 with the stochastic Round(.), Sec. III-A): 0 = round to nearest even
  int sr;
  unsigned sr_seed_lo, sr_seed_hi;   // the 64-bit seed
  unsigned sr_key0;                  // stream key of elements whose index is below 2^32 (computed on the host)
  int sr_wide;                       // 1: the tensor has 2^32 elements or more (keys are derived per element)
  int act;                           // mq_act applied to every element before quantization (channel-fastest source only; 0: none)
  int line;                          // 1: line blocks (one scale per row and 32 channels; the sc strides are per row), 0: 32 x 32 tiles
  unsigned int* status;              // device status word: set when a bounded wait gives up
  // test hooks of the TMA kernel's abort path: polls a barrier wait may take (0: the default limit), and 1 = the loader
  // issues no copies, so that every wait on them runs out
  unsigned wait_limit;
  int debug_skip_loads;
  // the paper's own format on the whole-line kernel (launch_quantize_ts_tma): where Eq. 4 takes max|X| from, and the
  // tensor's statistics buffer (T_scale is written to [0])
  const float* ts_amax;
  float* ts_stats;
  int packed6;        // 1: 6-bit codes leave packed, 16 codes in 12 bytes (out strides stay in elements)
  int ts_track_max;   // 1: the kernel also collects max|X| into ts_stats[1] (maximum supplied from outside: the tensor is read once)
};
// invertible 32-bit mixer (xor-shift, odd multiply, twice, xor-shift) behind the per-element draws
__host__ __device__ __forceinline__ unsigned sr_mix32(unsigned x) {
  x ^= x >> 16; x *= 0x7FEB352Du; x ^= x >> 15; x *= 0x846CA68Bu; x ^= x >> 16;
  return x;
}
cudaError_t launch_quantize(const QuantArgs& a, cudaStream_t s);
// The paper's own format (fp32 tensor scale, E4M3 scale per 16 x 16 block, E2M1 elements; mq_quantize_ts.cu).  stats: device, two
// floats (T_scale, max|X|); amax_in: device fp32 that Eq. 4 takes its maximum from, or null for the tensor's own.
cudaError_t launch_quantize_ts(const QuantArgs& a, const float* amax_in, float* stats, cudaStream_t s);
// Second pass of that quantizer on the whole-line TMA kernel (NCHW / OIHW source with 16-byte rows): true if the tensor qualifies
bool quantize_ts_tma_eligible(const QuantArgs& a);
cudaError_t launch_quantize_ts_tma(const QuantArgs& a, const float* amax_src, float* stats, cudaStream_t s, bool track_max = false);

struct Im2colArgs {
  const uint8_t* codes;
  const uint8_t* scales;
  uint8_t* out_codes;
  uint8_t* out_scales;
  Geom g;
  int fmt;
  int line;   // 1: line blocks (scales per sample instead of per 32 samples)
  int ts16;   // 1: 16 x 16 blocks (scales per 16 samples and 16 channels)
};
cudaError_t launch_im2col(const Im2colArgs& a, cudaStream_t s);

struct ConvArgs {
  Geom g;
  const uint8_t* a_codes;  // first operand of the call (fwd: X, bwd_data: W, bwd_weight: X)
  const uint8_t* a_scales;
  const uint8_t* b_codes;  // second operand (fwd: W, bwd_data: G_Y, bwd_weight: G_Y)
  const uint8_t* b_scales;
  int fmt_a, fmt_b;
  float* out;
  int out_layout;
  void* workspace;
  size_t ws_bytes;
  int line;   // 1: both operands carry line-block scales (one per row), forward GEMM only
  int ts16;   // 1: both operands are in the paper's own format: E4M3 scales per 16 x 16 block and a tensor scale each
  const float* a_tscale;   // device: T_scale of the first / second operand (ts16)
  const float* b_tscale;
};
// CUDA-core implicit-GEMM kernels: every shape, every format pair.
cudaError_t launch_conv_generic(int op, const ConvArgs& a, cudaStream_t s);
size_t conv_generic_workspace(int op, const Geom& g);
int conv_generic_bwd_weight_splits(const Geom& g);

// ---- device helpers --------------------------------------------------------------------------
#ifdef __CUDACC__

// 2^(code-127) as fp32 (code 0 gives the subnormal 2^-127)
__device__ __forceinline__ float e8m0_to_float(unsigned code) {
  return code == 0 ? __uint_as_float(0x00400000u) : __uint_as_float(code << 23);
}

// Exact decode of 8 consecutive codes (K- or MN-contiguous in memory) to fp32, times `scale`.
template <int FMT>
__device__ __forceinline__ void decode8(const uint8_t* codes_base, long long elem_off, float scale, float* out, int fmt8 = FMT) {
  // FMT: MQ_E2M1 (packed nibbles) or any other value for the one-byte-per-code formats, whose actual format is fmt8
  if (FMT == MQ_E2M1) {
    uint32_t v = *reinterpret_cast<const uint32_t*>(codes_base + (elem_off >> 1));
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      __half2_raw h = __nv_cvt_fp4x2_to_halfraw2((__nv_fp4x2_storage_t)((v >> (8 * i)) & 0xFF), __NV_E2M1);
      float2 f = __half22float2(*reinterpret_cast<__half2*>(&h));
      out[2 * i] = f.x * scale;
      out[2 * i + 1] = f.y * scale;
    }
  } else {
    uint2 v = *reinterpret_cast<const uint2*>(codes_base + elem_off);
    uint32_t w[2] = {v.x, v.y};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      unsigned short pair = (unsigned short)((w[i >> 1] >> (16 * (i & 1))) & 0xFFFF);
      __half2_raw h;
      if (fmt8 == MQ_E4M3) h = __nv_cvt_fp8x2_to_halfraw2((__nv_fp8x2_storage_t)pair, __NV_E4M3);
      else if (fmt8 == MQ_E5M2) h = __nv_cvt_fp8x2_to_halfraw2((__nv_fp8x2_storage_t)pair, __NV_E5M2);
      else if (fmt8 == MQ_E3M2) h = __nv_cvt_fp6x2_to_halfraw2((__nv_fp6x2_storage_t)pair, __NV_E3M2);
      else h = __nv_cvt_fp6x2_to_halfraw2((__nv_fp6x2_storage_t)pair, __NV_E2M3);
      float2 f = __half22float2(*reinterpret_cast<__half2*>(&h));
      out[2 * i] = f.x * scale;
      out[2 * i + 1] = f.y * scale;
    }
  }
}

// ---- quantization arithmetic shared by the quantizer kernels and the quantizing GEMM epilogue (Eq. 5-6, E8M0 form) ----
template <int FMT>
__device__ __forceinline__ unsigned encode2(float lo, float hi) {
  // two elements -> two codes (lo in the low byte / nibble), round-to-nearest-even, saturating
  if (FMT == MQ_E2M1) {
    return (unsigned)__nv_cvt_float2_to_fp4x2(make_float2(lo, hi), __NV_E2M1, cudaRoundNearest);
  } else if (FMT == MQ_E3M2 || FMT == MQ_E2M3) {
    // two 6-bit codes, each in the low six bits of its byte (the container the tensor core reads)
    return (unsigned)__nv_cvt_float2_to_fp6x2(make_float2(lo, hi), FMT == MQ_E3M2 ? __NV_E3M2 : __NV_E2M3, cudaRoundNearest);
  } else {
    return (unsigned)__nv_cvt_float2_to_fp8x2(make_float2(lo, hi), __NV_SATFINITE, FMT == MQ_E4M3 ? __NV_E4M3 : __NV_E5M2);
  }
}

// x / den of Eq. 6 (den = Scale_b x T_scale, or 0 for an all-zero block / tensor: the element is then a signed zero).  A zero
// numerator would send __fdiv_rn down its slow path (a call that the whole warp waits for - post-ReLU tensors are half
// zeros: measured 2x on the quantizing epilogue), so zeros divide a stand-in and keep their sign; the quotient of every
// other value is the IEEE one.
__device__ __forceinline__ float ts_div(float x, float den) {
  const bool z = x == 0.f || !(den > 0.f);
  const float q = __fdiv_rn(z ? 1.f : x, z ? 1.f : den);
  return z ? copysignf(0.f, x) : q;
}

// activation of the quantizing producer epilogue (mq_act), evaluated in fp32
__device__ __forceinline__ float mx_activation(float y, int act) {
  if (act == MQ_ACT_RELU) return fmaxf(y, 0.f);
  if (act == MQ_ACT_SILU) return __fdividef(y, 1.f + __expf(-y));
  return y;
}

__device__ __forceinline__ int scale_code_of(unsigned amax_bits, int emax) {
  // floor(log2 amax) = biased exponent - 127 for normal amax; subnormal / zero amax clamps to 0
  const int e = (int)(amax_bits >> 23) - emax;
  return min(max(e, 0), 254);
}

// 2^(127 - code) as a normal fp32 number: code = clamp(E - emax, 0, 254) with E <= 254 and emax >= 2, so
// 127 - code lies in [-125, 127].  x * 2^(127 - code) is then exact (|result| < 2^(emax + 1)) except where it
// underflows below 2^-126, far under half of the smallest element step, where it rounds to zero either way.
__device__ __forceinline__ float scale_factor(int code) { return __uint_as_float((unsigned)(254 - code) << 23); }

// Stochastic Round(.) of Eq. 6 (Sec. III-A: the gradient's rounding).  x is the scaled element, idx its index in the
// logical NCHW / OIHW tensor.  The element's draw is 32 bits of a counter-based generator keyed by (seed, idx);
// u = (top 23 bits + 1/2) / 2^23.  With lo <= |x| < hi neighbours on the format's grid, the result is hi when
// u < (|x| - lo) / (hi - lo), else lo -- returned as a float that lies on the grid, so the round-to-nearest
// conversion that follows is exact.  Everything below is exact in fp32: |x| / step has at most 24 significant bits,
// its fractional part and (23-bit draw + 1/2) likewise.  Magnitudes at or beyond the largest one are left to the
// conversion's saturation.
// lo: low word of the element's index; key: the stream key of its high word (sr_key)
template <int FMT>
__device__ __forceinline__ float sr_value(float x, unsigned lo, unsigned key) {
  constexpr int M = (FMT == MQ_E4M3 || FMT == MQ_E2M3) ? 3 : (FMT == MQ_E2M1 ? 1 : 2);                      // mantissa bits
  constexpr int EMIN = FMT == MQ_E4M3 ? -6 : (FMT == MQ_E5M2 ? -14 : (FMT == MQ_E3M2 ? -2 : 0));           // smallest normal exponent
  const unsigned b = __float_as_uint(x) & 0x7fffffffu;       // |x|; patterns of non-negative floats order like their values
  const unsigned rn = ~sr_mix32(lo ^ key);                   // the draw's complement: top 23 bits = 2^23 - 1 - draw
  // normal range of the format: the grid keeps M mantissa bits of the fp32 pattern.  The dropped field f (23 - M bits) is the
  // fraction of a step in units of 2^-(23 - M): up iff f * 2^M > draw, i.e. iff f + (2^(23 - M) - 1 - (draw >> M)) carries
  // out of the field - so one addition on the pattern decides and steps (the carry walks into the exponent at a binade's end).
  constexpr unsigned MASK = (1u << (23 - M)) - 1u;
  const unsigned q_norm = (b + (rn >> (9 + M))) & ~MASK;
  // below it the step is the constant 2^(EMIN - M): t = |x| / step < 2^M, up iff frac(t) > u = (draw + 1/2) / 2^23, i.e. the result
  // is ceil(t + (1 - u)) - 1.  1 - u = (2^23 - 1 - draw) 2^-23 + 2^-24 is exact; rounding the sum up, and then to an integer by an
  // addition of 2^23 rounded up, keeps the ceiling.
  const float t = __uint_as_float(b) * __uint_as_float((unsigned)(127 + M - EMIN) << 23);
  const float w = __uint_as_float(0x3F800000u | (rn >> 9)) - __uint_as_float(0x3F7FFFFFu);
  const float n = __fadd_ru(__fadd_ru(t, w), 8388608.f) - 8388609.f;
  const unsigned q_sub = __float_as_uint(n * __uint_as_float((unsigned)(127 + EMIN - M) << 23));
  // Beyond the largest magnitude the conversion saturates.  The comparison is one of floats because a NaN has to take the second
  // branch, whose arithmetic keeps it one: the addition above would carry its pattern into the sign, that is to -0.
  const unsigned q = __uint_as_float(b) >= __uint_as_float((unsigned)(127 + EMIN) << 23) ? q_norm : q_sub;
  return __uint_as_float(q | (__float_as_uint(x) & 0x80000000u));
}

// Stream key of an element from the high word of its index; tensors below 2^32 elements (a.sr_wide == 0, uniform)
// take the key computed on the host.
__device__ __forceinline__ unsigned sr_key(const QuantArgs& a, long long idx) {
  if (!a.sr_wide) return a.sr_key0;
  return sr_mix32(a.sr_seed_lo ^ sr_mix32(a.sr_seed_hi ^ sr_mix32((unsigned)((unsigned long long)idx >> 32))));
}

// ---- elements of the paper's own format (Eq. 6: Round(x / den), den = Scale_b x T_scale) ---------------------------------
// The quotient is an IEEE division, but it only decides which of E2M1's eight magnitudes comes out, so the division itself is
// rarely needed: q' = x * (1 / den) is within 2.5 units in the last place of it, and unless q' lies within four units of a
// decision threshold both round alike.  The few elements for which that cannot be said (one in 10^5; all of a block whose
// denominator is so extreme that the bound on q' does not hold) are divided.  An IEEE division costs a dozen instructions and
// a branch per element, the check three (256 channels 28x28, N = 256: 72 -> 61 us, stochastic 185 -> 106 us).
struct TsDen {
  float den, inv;   // den 0: the block encodes to signed zeros
  unsigned sure;    // 0: every element takes the division
};
__device__ __forceinline__ TsDen ts_den(float den) {
  TsDen d;
  d.den = den;
  const bool in_range = den >= 7.9e-31f && den <= 1.2e30f;    // 2^-100 .. 2^100
  d.inv = in_range ? __frcp_rn(den) : 0.f;
  d.sure = (in_range || !(den > 0.f)) ? 0xffffffffu : 0u;
  return d;
}
// fmaxf / fminf that keep a NaN
__device__ __forceinline__ float max_nan(float a, float b) { float r; asm("max.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b)); return r; }
__device__ __forceinline__ float min_nan(float a, float b) { float r; asm("min.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b)); return r; }
// One element by the definition.  lo, key: as sr_value's
template <bool SR>
__device__ __forceinline__ unsigned ts_code_by_division(float x, float den, unsigned lo, unsigned key) {
  float q = ts_div(x, den);
  if (SR && den > 0.f) q = sr_value<MQ_E2M1>(q, lo, key);
  return encode2<MQ_E2M1>(q, 0.f) & 0xFu;
}
// Eight elements of neighbouring channels -> their codes, element 0 in the low nibble.  e0 (SR): element 0's index in the logical
// tensor, whose channels are a.P elements apart.  A NaN product - of a NaN, or of an infinity and the 0 of a block that encodes to
// zeros - says nothing either: the window tests let it through to the division.
template <bool SR>
__device__ __forceinline__ unsigned ts_codes8(const float* x, const TsDen& d, const QuantArgs& a, long long e0) {
  unsigned word = 0, sure = d.sure;
  if (!SR) {
    // thresholds of round-to-nearest are 0.25, 0.75, 1.25, 1.75, 2.5, 3.5 and 5: patterns whose low 21 bits are zero (and a
    // NaN's, all ones, is one short of it)
#pragma unroll
    for (int k = 0; k < 8; k += 2) {
      const float q0 = x[k] * d.inv, q1 = x[k + 1] * d.inv;
      sure = min(sure, (__float_as_uint(max_nan(fabsf(q0), 0.24f)) + 4u) << 11);
      sure = min(sure, (__float_as_uint(max_nan(fabsf(q1), 0.24f)) + 4u) << 11);
      word |= encode2<MQ_E2M1>(q0, q1) << (4 * k);
    }
    if (sure >= (8u << 11)) return word;
  } else {
    // As in sr_value, one addition on the pattern of q' decides and steps; below 1 the pattern of q' + 1, two codes down, whose
    // last place is 2^-22 of the step 0.5 - the sum's low 22 bits tell how far the decision is (window: 2.5 units of q', one of
    // the addition and one of the draw's finer bits, rounded up to 8)
    const unsigned lo0 = (unsigned)e0;
    unsigned key = a.sr_key0;
    if (a.sr_wide) {   // (eight channels across which the index's high word advances have two keys: by division)
      key = sr_key(a, e0);
      if ((unsigned long long)(e0 + 7ll * a.P) >> 32 != (unsigned long long)e0 >> 32) sure = 0;
    }
    float total = 0.f;     // NaN if any product is (a float addition, on a pipe that this loop leaves idle)
#pragma unroll
    for (int k = 7; k >= 0; --k) {
      const unsigned rn = ~sr_mix32((lo0 + (unsigned)k * (unsigned)a.P) ^ key);
      const float q = min_nan(fabsf(x[k]) * d.inv, 6.f);
      total += q;
      const bool below = q < 1.f;
      const unsigned sum = __float_as_uint(below ? q + 1.f : q) + (rn >> 10) + (below ? 0u - (254u << 22) : 0u - (252u << 22));
      sure = min(sure, (sum + 8u) << 10);
      word = __funnelshift_l((sum << 6) | (__float_as_uint(x[k]) & 0x80000000u), word, 4);
    }
    if (sure >= (16u << 10) && total == total) return word;
  }
#pragma unroll 1
  for (int k = 0; k < 8; ++k) {
    float xk = x[0];
#pragma unroll
    for (int j = 1; j < 8; ++j) xk = j == k ? x[j] : xk;
    const long long e = e0 + (long long)k * a.P;
    word = (word & ~(0xFu << (4 * k))) | (ts_code_by_division<SR>(xk, d.den, (unsigned)e, SR ? sr_key(a, e) : 0u) << (4 * k));
  }
  return word;
}

#endif  // __CUDACC__

// ---- programmatic dependent launch --------------------------------------------------------------------------
// Kernels of this library are launched with programmatic stream serialization: a kernel may be scheduled while its
// predecessor in the stream is still draining, and executes pdl_wait() (griddepcontrol.wait: returns once the
// predecessor grid has completed and its writes are visible) before its first access to global memory.  Every
// kernel waits, so completion is transitive along the stream.  MQ_NO_PDL=1 launches them plainly.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
bool pdl_enabled();
template <typename... KArgs, typename... Args>
cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr; cfg.numAttrs = pdl_enabled() ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}
// the same with thread-block clusters of `cluster_x` consecutive blocks (grid.x a multiple of it)
template <typename... KArgs, typename... Args>
cudaError_t launch_pdl_cluster(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, unsigned cluster_x, Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = cluster_x; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr; cfg.numAttrs = pdl_enabled() ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

}  // namespace mq
