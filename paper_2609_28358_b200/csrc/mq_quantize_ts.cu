// Quantizer of the paper's own number format (Sec. III-A): an fp32 scale per tensor (Eq. 4), an E4M3 scale per block
// (Eq. 5), E2M1 elements (Eq. 6), on 16 x 16 square blocks over the two axes Sec. IV-B names for each tensor - the
// square's side set to the tensor core's finest scale granularity (16 elements), the paper's own 8 x 8 being below it.
//
// Two passes when the tensor's own maximum is wanted (Eq. 4 needs max|X| before any element can be scaled): a reduction leaves
// max|X| in the tensor's statistics buffer, the quantizer then reads it.  With the maximum supplied from outside (statistics of
// earlier batches, Sec. VII-B) nothing has to wait for this tensor's maximum: the tensor is read ONCE, the quantizer collecting
// max|X| for the next step from the block maxima it forms anyway (tensors of less than 2^17 elements, for which the memset
// that an atomic maximum starts from costs what the reduction does, keep the two launches).
//
// Every operation of Eq. 4-6 is one IEEE single-precision operation, in the order written (division = __fdiv_rn,
// products = __fmul_rn): the roundings decide integer codes, so nothing here may be contracted.  Eq. 6's quotient decides no more than
// which of eight magnitudes comes out: ts_codes8 multiplies by the reciprocal and divides only where that product does not say.
// CastE4M3 and Round(.) are the hardware's round-to-nearest-even, saturating conversions.
//
// quantize_ts_kernel: one warp per (16 x 16 block, 8 consecutive positions).  Lane (r, h) = (lane >> 1, lane & 1) owns
// row r, channels 8 h .. 8 h + 7 of the block at the 8 positions: 64 values.  From an NCHW source the 8 positions of a
// (row, channel) are 32 contiguous bytes (two 128-bit loads); from a channel-fastest source the 8 channels are.  Block
// maxima are warp reductions (one per position), a lane's 8 codes leave as one 32-bit store, lane 0 writes the block's
// scale bytes.
#include "mq_internal.cuh"
#include "mq_tcgen05.cuh"   // cluster barrier and addresses

namespace mq {
namespace {

// max|x| over this thread's share of n floats (a dense array, whichever the source's order).  act: mq_act applied to every element
// first (the two-launch route of the quantizing epilogue), 0 = none.  Four 128-bit loads in flight.
__device__ __forceinline__ float amax_share(const float* __restrict__ src, long long n, long long t0, long long stride, int act) {
  float m = 0.f;
  auto take = [&](float4 v) {
    if (act) { v.x = mx_activation(v.x, act); v.y = mx_activation(v.y, act); v.z = mx_activation(v.z, act); v.w = mx_activation(v.w, act); }
    m = fmaxf(fmaxf(m, fmaxf(fabsf(v.x), fabsf(v.y))), fmaxf(fabsf(v.z), fabsf(v.w)));
  };
  const long long n4 = (reinterpret_cast<uintptr_t>(src) & 15) == 0 ? n >> 2 : 0;
  const float4* s4 = reinterpret_cast<const float4*>(src);
  long long i = t0;
  for (; i + 3 * stride < n4; i += 4 * stride) {
    const float4 v0 = __ldg(s4 + i), v1 = __ldg(s4 + i + stride), v2 = __ldg(s4 + i + 2 * stride), v3 = __ldg(s4 + i + 3 * stride);
    take(v0); take(v1); take(v2); take(v3);
  }
  for (; i < n4; i += stride) take(__ldg(s4 + i));
  for (i = 4 * n4 + t0; i < n; i += stride) m = fmaxf(m, fabsf(act ? mx_activation(__ldg(src + i), act) : __ldg(src + i)));
  return m;
}
__global__ void __launch_bounds__(256) tensor_amax_kernel(const float* __restrict__ src, long long n, unsigned* __restrict__ amax_bits, int act) {
  pdl_wait();
  const float m = amax_share(src, n, (long long)blockIdx.x * blockDim.x + threadIdx.x, (long long)gridDim.x * blockDim.x, act);
  const unsigned w = __reduce_max_sync(0xffffffffu, __float_as_uint(m));    // bit patterns of non-negative floats order like the values
  if ((threadIdx.x & 31) == 0 && w != 0) atomicMax(amax_bits, w);
}
// The same for tensors of at most AMAX_CLUSTER_MOST floats by one cluster of eight blocks, which combine their maxima through
// distributed shared memory and WRITE the result: no memset before it and no atomics (weights of 256 -> 256 channels, 3x3: what
// comes before the quantizer takes one launch of about 4 us instead of a memset, its gap and a launch).
constexpr int AMAX_CLUSTER = 8, AMAX_THREADS = 1024;
constexpr long long AMAX_CLUSTER_MOST = 1ll << 20;
__global__ void __launch_bounds__(AMAX_THREADS) tensor_amax_cluster_kernel(const float* __restrict__ src, long long n, unsigned* __restrict__ amax_bits, int act) {
  __shared__ unsigned warp_max[AMAX_THREADS / 32];
  __shared__ unsigned block_max;
  pdl_wait();
  const float m = amax_share(src, n, (long long)blockIdx.x * AMAX_THREADS + threadIdx.x, (long long)AMAX_CLUSTER * AMAX_THREADS, act);
  const unsigned w = __reduce_max_sync(0xffffffffu, __float_as_uint(m));
  if ((threadIdx.x & 31) == 0) warp_max[threadIdx.x >> 5] = w;
  __syncthreads();
  if (threadIdx.x < 32) {
    const unsigned b = __reduce_max_sync(0xffffffffu, warp_max[threadIdx.x]);
    if (threadIdx.x == 0) block_max = b;
  }
  __syncwarp();
  tc::cluster_sync_all();
  if (blockIdx.x == 0 && threadIdx.x < 32) {
    unsigned v = 0;
    if (threadIdx.x < AMAX_CLUSTER) asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(tc::cluster_addr_of(&block_max, threadIdx.x)));
    v = __reduce_max_sync(0xffffffffu, v);
    if (threadIdx.x == 0) *amax_bits = v;
  }
  __syncwarp();
  tc::cluster_sync_all();   // no block leaves while its shared memory may be read
}

__device__ __forceinline__ float e4m3_value(unsigned code) {
  const __half_raw h = __nv_cvt_fp8_to_halfraw((__nv_fp8_storage_t)code, __NV_E4M3);
  return __half2float(*reinterpret_cast<const __half*>(&h));
}

// Scale byte and denominator of a block from the bit pattern of its maximum (Eq. 5)
__device__ __forceinline__ TsDen ts_block_den(unsigned bmax_bits, float tscale, float t6, unsigned* scale) {
  const float bmax = __uint_as_float(bmax_bits);
  unsigned sc = 0;
  if (bmax > 0.f && tscale > 0.f) sc = (unsigned)__nv_cvt_float_to_fp8(__fdiv_rn(bmax, t6), __NV_SATFINITE, __NV_E4M3) & 0x7Fu;
  const float bscale = e4m3_value(sc);
  *scale = sc;
  return ts_den((bscale > 0.f && tscale > 0.f) ? __fmul_rn(bscale, tscale) : 0.f);
}

// OIHW / NCHW source with few positions (the taps of a weight tensor): the 16 channels x P positions of a row are one run of
// 16 P floats.  A block brings the 16 runs of a (row block, channel block) into shared memory as whole lines - read 8 positions at a
// time straight from global memory they are one 4-byte load per element, P elements apart - and its warps then take a position
// each, lane (r, h) = (row, channel half) as in quantize_ts_kernel.  256 -> 256 channels, 3x3, with its
// maximum: 16.4 -> 8.2 us.
constexpr int TS_FEW = 40;      // most positions (43 KB of shared memory)
__device__ __host__ constexpr int ts_few_stride(int P) { return 16 * P + ((33 - 16 * P % 32) & 31); }   // floats per row, 1 modulo 32: rows start in different banks
template <bool SR>
__global__ void __launch_bounds__(256) quantize_ts_few_kernel(QuantArgs a, const float* __restrict__ amax_src, float* __restrict__ stats, int Cb, int track) {
  extern __shared__ float few[];
  pdl_wait();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const float tscale = __fdiv_rn(*amax_src, __fmul_rn(448.0f, 6.0f));                        // Eq. 4
  if (blockIdx.x == 0 && threadIdx.x == 0) stats[0] = tscale;
  const float t6 = __fmul_rn(tscale, 6.0f);
  const int rb = (int)(blockIdx.x / (unsigned)Cb), cb = (int)(blockIdx.x - (unsigned)rb * (unsigned)Cb);
  const int stride = ts_few_stride(a.P), run = 16 * a.P, valid = min(16, a.C - cb * 16) * a.P;   // (valid <= 0: padded channels only)
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const int row = 2 * warp + i, r = rb * 16 + row;
    const float* src = a.src + ((long long)r * a.C + cb * 16) * a.P;
    for (int k = lane; k < run; k += 32) few[row * stride + k] = (r < a.R && k < valid) ? __ldg(src + k) : 0.f;
  }
  __syncthreads();
  const int r_l = lane >> 1, h = lane & 1, r = rb * 16 + r_l, c0 = cb * 16 + 8 * h;
  unsigned own_max = 0;
#pragma unroll 1
  for (int p = warp; p < a.P; p += 8) {
    float x[8], m = 0.f;
#pragma unroll
    for (int k = 0; k < 8; ++k) { x[k] = few[r_l * stride + (8 * h + k) * a.P + p]; m = fmaxf(m, fabsf(x[k])); }
    const unsigned bmax = __reduce_max_sync(0xffffffffu, __float_as_uint(m));
    own_max = max(own_max, bmax);
    unsigned sc;
    const TsDen den = ts_block_den(bmax, tscale, t6, &sc);
    if (lane == 0) a.scales[(long long)p * a.sc_stride_p + (long long)rb * a.sc_stride_r + cb] = (uint8_t)sc;
    const unsigned word = ts_codes8<SR>(x, den, a, ((long long)r * a.C + c0) * a.P + p);     // Eq. 6
    if (r < a.R) *reinterpret_cast<unsigned*>(a.codes + (((long long)p * a.out_stride_p + (long long)r * a.out_stride_r + c0) >> 1)) = word;
  }
  if (track && lane == 0 && own_max != 0) atomicMax(reinterpret_cast<unsigned*>(stats + 1), own_max);   // (own_max is the warp's)
}

// stats: [0] T_scale (written here), [1] max|X| of this tensor (written by the first pass, or, track, collected here on top of
// zero); amax_src: where Eq. 4 takes its maximum from: &stats[1], or the caller's value
template <bool SR>
__global__ void __launch_bounds__(256) quantize_ts_kernel(QuantArgs a, const float* __restrict__ amax_src, float* __restrict__ stats, int Rb, int Cb,
                                                          unsigned n_pstrips, unsigned n_items, int vec, int track) {
  pdl_wait();
  const int lane = threadIdx.x & 31;
  const int r_l = lane >> 1, h = lane & 1;
  const float tscale = __fdiv_rn(*amax_src, __fmul_rn(448.0f, 6.0f));                        // Eq. 4
  if (blockIdx.x == 0 && threadIdx.x == 0) stats[0] = tscale;
  const float t6 = __fmul_rn(tscale, 6.0f);
  unsigned own_max = 0;
#pragma unroll 1
  for (unsigned it = blockIdx.x * 8u + (threadIdx.x >> 5); it < n_items; it += gridDim.x * 8u) {
    // position strip fastest, then channel block, then row block
    const unsigned ps = it % n_pstrips; const unsigned u = it / n_pstrips;
    const int cb = (int)(u % (unsigned)Cb), rb = (int)(u / (unsigned)Cb);
    const int p0 = (int)ps * 8, r = rb * 16 + r_l, c0 = cb * 16 + 8 * h;
    float v[8][8];   // [channel][position]
#pragma unroll
    for (int k = 0; k < 8; ++k)
#pragma unroll
      for (int j = 0; j < 8; ++j) v[k][j] = 0.f;
    if (r < a.R) {
      if (a.src_stride_r == 0) {   // NCHW / OIHW: element (p, r, c) at (r C + c) P + p
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          if (c0 + k < a.C) {
            const float* q = a.src + ((long long)r * a.C + c0 + k) * a.P + p0;
            if (vec && p0 + 8 <= a.P) {
              const float4 lo = __ldg(reinterpret_cast<const float4*>(q)), hi = __ldg(reinterpret_cast<const float4*>(q) + 1);
              v[k][0] = lo.x; v[k][1] = lo.y; v[k][2] = lo.z; v[k][3] = lo.w; v[k][4] = hi.x; v[k][5] = hi.y; v[k][6] = hi.z; v[k][7] = hi.w;
            } else {
#pragma unroll
              for (int j = 0; j < 8; ++j) if (p0 + j < a.P) v[k][j] = __ldg(q + j);
            }
          }
        }
      } else {                     // channel-fastest: element (p, r, c) at p stride_p + r stride_r + c
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          if (p0 + j < a.P) {
            const float* q = a.src + (long long)(p0 + j) * a.src_stride_p + (long long)r * a.src_stride_r + c0;
#pragma unroll
            for (int k = 0; k < 8; ++k) if (c0 + k < a.C) v[k][j] = a.act ? mx_activation(__ldg(q + k), a.act) : __ldg(q + k);
          }
        }
      }
    }
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      float m = 0.f;
#pragma unroll
      for (int k = 0; k < 8; ++k) m = fmaxf(m, fabsf(v[k][j]));
      const unsigned bmax = __reduce_max_sync(0xffffffffu, __float_as_uint(m));
      own_max = max(own_max, bmax);
      unsigned sc;
      const TsDen den = ts_block_den(bmax, tscale, t6, &sc);
      const bool p_ok = p0 + j < a.P;
      if (lane == 0 && p_ok) a.scales[(long long)(p0 + j) * a.sc_stride_p + (long long)rb * a.sc_stride_r + cb] = (uint8_t)sc;
      float x[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) x[k] = v[k][j];
      const unsigned word = ts_codes8<SR>(x, den, a, ((long long)r * a.C + c0) * a.P + p0 + j);     // Eq. 6
      if (p_ok && r < a.R) {
        const long long e = (long long)(p0 + j) * a.out_stride_p + (long long)r * a.out_stride_r + c0;
        *reinterpret_cast<unsigned*>(a.codes + (e >> 1)) = word;
      }
    }
  }
  if (track && lane == 0 && own_max != 0) atomicMax(reinterpret_cast<unsigned*>(stats + 1), own_max);   // (own_max is the warp's)
}

}  // namespace

// stats: device, two floats (T_scale, max|X|).  amax_in: device fp32 to take Eq. 4's maximum from, or null for the
// tensor's own.
cudaError_t launch_quantize_ts(const QuantArgs& a, const float* amax_in, float* stats, cudaStream_t s) {
  const long long n = (long long)a.P * a.R * a.C;
  if (a.act && a.src_stride_r == 0) return cudaErrorInvalidValue;   // the activation rides on the channel-fastest source only
  const int Rb = (a.R + 15) / 16, Cb = a.Cp / 16;
  const long long n_pstrips = (a.P + 7) / 8, n_items = n_pstrips * Rb * Cb;
  if (n_items <= 0 || n_items > 0xffffffffLL) return cudaErrorInvalidValue;
  const bool few = a.src_stride_r == 0 && a.P <= TS_FEW && a.P % 4 != 0 && (long long)Rb * Cb <= 0x7fffffffLL;
  const bool whole_lines = quantize_ts_tma_eligible(a);
  // maximum supplied from outside: ONE pass - the quantizer collects this tensor's own maximum for the next step while it works
  // (MQ_QUANT_TS_TWO_PASS=1 keeps the separate reduction)
  const bool one_pass = amax_in && (whole_lines || n >= (1ll << 17)) && !MQ_ENV("MQ_QUANT_TS_TWO_PASS", 0);
  const bool cluster = !one_pass && n <= AMAX_CLUSTER_MOST;
  cudaError_t e = cudaSuccess;
  if (!cluster) e = cudaMemsetAsync(stats + 1, 0, sizeof(float), s);     // an atomic maximum starts from zero
  if (e != cudaSuccess) return e;
  unsigned* own = reinterpret_cast<unsigned*>(stats + 1);
  if (!one_pass) {   // the source of either layout is a dense array of n floats
    long long blocks = (n / 4 + 255) / 256;
    if (blocks > (long long)sm_count() * 8) blocks = (long long)sm_count() * 8;
    if (blocks < 1) blocks = 1;
    e = cluster ? launch_pdl_cluster(tensor_amax_cluster_kernel, dim3(AMAX_CLUSTER), dim3(AMAX_THREADS), 0, s, AMAX_CLUSTER, a.src, n, own, a.act)
                : launch_pdl(tensor_amax_kernel, dim3((unsigned)blocks), dim3(256), 0, s, a.src, n, own, a.act);
    if (e != cudaSuccess) return e;
    count_launches(1);
  }
  count_launches(1);
  const float* amax_src = amax_in ? amax_in : stats + 1;
  // large NCHW / OIHW tensors with 16-byte rows: the whole-line TMA kernel (items of 32 positions x 32 rows x 32 channels = 4 blocks per position)
  if (whole_lines) return launch_quantize_ts_tma(a, amax_src, stats, s, one_pass);
  if (few) {
    const size_t smem = (size_t)16 * ts_few_stride(a.P) * sizeof(float);
    return launch_pdl(a.sr ? quantize_ts_few_kernel<true> : quantize_ts_few_kernel<false>, dim3((unsigned)(Rb * Cb)), dim3(256), smem, s, a, amax_src, stats, Cb,
                      one_pass ? 1 : 0);
  }
  long long qb = (n_items + 7) / 8;
  if (qb > (long long)sm_count() * 32) qb = (long long)sm_count() * 32;
  const int vec = (a.P % 4 == 0 && (reinterpret_cast<uintptr_t>(a.src) & 15) == 0) ? 1 : 0;
  return launch_pdl(a.sr ? quantize_ts_kernel<true> : quantize_ts_kernel<false>, dim3((unsigned)qb), dim3(256), 0, s, a, amax_src, stats, Rb, Cb, (unsigned)n_pstrips,
                    (unsigned)n_items, vec, one_pass ? 1 : 0);
}

}  // namespace mq
