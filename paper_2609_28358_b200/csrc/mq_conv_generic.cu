// CUDA-core implicit-GEMM kernels for the three block-scaled convolution GEMMs (Sec. II-C, IV-B,
// Eq. 7).  They accept every shape and every element-format pair and serve the shapes the
// tensor-core kernels do not cover (thin channel counts, odd geometry).  Operands are decoded
// exactly (code -> fp16 -> fp32, times the tile's power-of-two scale) into shared memory, one
// 32-element MX block of K per step, and accumulated in fp32.
//
//   fwd        : M = (ho,wo,n)   N = co           K = (kh,kw | ci)   A = X gathered, B = W     both K-contiguous
//   bwd_data   : M = (h,w,n)     N = ci           K = (kh,kw | co)   A = G_Y gathered (K-contiguous), B = W (N-contiguous)
//   bwd_weight : M = co          N = (kh,kw,ci)   K = (ho,wo | n)    A = G_Y, B = X gathered   both MN-contiguous
#include "mq_conv_tc.cuh"

namespace mq {
namespace {

constexpr int TM = 64, TN = 64, TK = 32, GT = 256, PADF = 4;

struct Tiles {
  alignas(16) float As[TK][TM + PADF];
  alignas(16) float Bs[TK][TN + PADF];
};

__device__ __forceinline__ void store_kmajor(float (*S)[TM + PADF], int row, int kq, const float* v) {
#pragma unroll
  for (int j = 0; j < 8; ++j) S[kq * 8 + j][row] = v[j];
}
__device__ __forceinline__ void store_mnmajor(float (*S)[TM + PADF], int k, int mq, const float* v) {
  *reinterpret_cast<float4*>(&S[k][mq * 8]) = make_float4(v[0], v[1], v[2], v[3]);
  *reinterpret_cast<float4*>(&S[k][mq * 8 + 4]) = make_float4(v[4], v[5], v[6], v[7]);
}
__device__ __forceinline__ void zero8(float* v) {
#pragma unroll
  for (int j = 0; j < 8; ++j) v[j] = 0.f;
}

// Scale of the 8 consecutive channels starting at channel c of row `row` at position `pos` of a stored tensor:
//   activation-like tensors ([pos][row][c], R rows): sc[(pos * RB + row_block) * CB + channel_block]
//   weights ([row][pos][c], P positions):            sc[(row_block * P + pos) * CB + channel_block]
// with 32 x 32 tiles (E8M0), line blocks (one row per block) or, ts16, 16 x 16 blocks whose E4M3 scale is multiplied by the
// tensor's fp32 scale t.
__device__ __forceinline__ float e4m3_to_float(unsigned code) {
  const __half_raw h = __nv_cvt_fp8_to_halfraw((__nv_fp8_storage_t)code, __NV_E4M3);
  return __half2float(*reinterpret_cast<const __half*>(&h));
}
__device__ __forceinline__ float act_scale(const ConvArgs& a, const uint8_t* sc, float t, long long pos, int row, int c, int R, int Cp) {
  if (a.ts16) return e4m3_to_float(sc[(pos * ((R + 15) >> 4) + (row >> 4)) * (Cp >> 4) + (c >> 4)]) * t;
  if (a.line) return e8m0_to_float(sc[(pos * R + row) * (Cp >> 5) + (c >> 5)]);
  return e8m0_to_float(sc[(pos * ((R + 31) >> 5) + (row >> 5)) * (Cp >> 5) + (c >> 5)]);
}
__device__ __forceinline__ float w_scale(const ConvArgs& a, const uint8_t* sc, float t, int row, int taps, int tap, int c, int Cp) {
  if (a.ts16) return e4m3_to_float(sc[((long long)(row >> 4) * taps + tap) * (Cp >> 4) + (c >> 4)]) * t;
  if (a.line) return e8m0_to_float(sc[((long long)row * taps + tap) * (Cp >> 5) + (c >> 5)]);
  return e8m0_to_float(sc[((long long)(row >> 5) * taps + tap) * (Cp >> 5) + (c >> 5)]);
}

__device__ __forceinline__ void mma_tile(const Tiles& sm, int ty, int tx, float acc[4][4]) {
#pragma unroll
  for (int k = 0; k < TK; ++k) {
    float4 a = *reinterpret_cast<const float4*>(&sm.As[k][ty * 4]);
    float4 b = *reinterpret_cast<const float4*>(&sm.Bs[k][tx * 4]);
    float av[4] = {a.x, a.y, a.z, a.w}, bv[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(av[i], bv[j], acc[i][j]);
  }
}

// ------------------------------------------------------------------------------------ forward
template <int FX, int FW>
__global__ void __launch_bounds__(GT) fwd_generic(ConvArgs a) {
  __shared__ Tiles sm;
  const Geom& g = a.g;
  const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15;
  const int row_l = tid >> 2, kq = tid & 3;
  const long long M = (long long)g.Ho * g.Wo * g.N;
  const long long m0 = (long long)blockIdx.x * TM;
  const int n0 = blockIdx.y * TN;
  const int taps = g.Kh * g.Kw;

  const long long m = m0 + row_l;
  const bool m_ok = m < M;
  int n = 0, wo = 0, ho = 0;
  if (m_ok) { n = (int)(m % g.N); long long q = m / g.N; wo = (int)(q % g.Wo); ho = (int)(q / g.Wo); }
  const int co = n0 + row_l;
  const bool co_ok = co < g.Cout;
  const float ta = a.ts16 ? *a.a_tscale : 1.f, tb = a.ts16 ? *a.b_tscale : 1.f;

  float acc[4][4] = {};
  for (int tap = 0; tap < taps; ++tap) {
    const int kh = tap / g.Kw, kw = tap - kh * g.Kw;
    const int h = ho * g.sh + kh - g.ph, w = wo * g.sw + kw - g.pw;
    const bool pix_ok = m_ok && h >= 0 && h < g.H && w >= 0 && w < g.W;
    const long long pix = (long long)h * g.W + w;
    for (int kb = 0; kb < g.Ct; ++kb) {
      float va[8], vb[8];
      if (pix_ok) {
        const float s = act_scale(a, a.a_scales, ta, pix, n, kb * 32 + kq * 8, g.N, g.Cp);
        decode8<FX>(a.a_codes, (pix * g.N + n) * g.Cp + kb * 32 + kq * 8, s, va, a.fmt_a);
      } else zero8(va);
      if (co_ok) {
        const float s = w_scale(a, a.b_scales, tb, co, taps, tap, kb * 32 + kq * 8, g.Cp);
        decode8<FW>(a.b_codes, ((long long)co * taps + tap) * g.Cp + kb * 32 + kq * 8, s, vb, a.fmt_b);
      } else zero8(vb);
      __syncthreads();
      store_kmajor(sm.As, row_l, kq, va);
      store_kmajor(sm.Bs, row_l, kq, vb);
      __syncthreads();
      mma_tile(sm, ty, tx, acc);
    }
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const long long mm = m0 + ty * 4 + i;
    if (mm >= M) continue;
    const int nn = (int)(mm % g.N); const long long q = mm / g.N;
    const int wwo = (int)(q % g.Wo), hho = (int)(q / g.Wo);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int c = n0 + tx * 4 + j;
      if (c >= g.Cout) continue;
      if (a.out_layout == MQ_NCHW) a.out[(((long long)nn * g.Cout + c) * g.Ho + hho) * g.Wo + wwo] = acc[i][j];
      else a.out[mm * g.Cout + c] = acc[i][j];
    }
  }
}

// --------------------------------------------------------------------------------- input gradient
template <int FW, int FG>
__global__ void __launch_bounds__(GT) bwd_data_generic(ConvArgs a) {
  __shared__ Tiles sm;
  const Geom& g = a.g;
  const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15;
  const int row_l = tid >> 2, kq = tid & 3;   // A units: (row, 8 consecutive k)
  const int k_l = tid >> 3, nq = tid & 7;     // B units: (k, 8 consecutive ci)
  const long long M = (long long)g.H * g.W * g.N;
  const long long m0 = (long long)blockIdx.x * TM;
  const int n0 = blockIdx.y * TN;
  const int taps = g.Kh * g.Kw;

  const long long m = m0 + row_l;
  const bool m_ok = m < M;
  int n = 0, w = 0, h = 0;
  if (m_ok) { n = (int)(m % g.N); long long q = m / g.N; w = (int)(q % g.W); h = (int)(q / g.W); }
  const int ci0 = n0 + nq * 8;
  const bool ci_ok = ci0 < g.Cp;
  const float ta = a.ts16 ? *a.a_tscale : 1.f, tb = a.ts16 ? *a.b_tscale : 1.f;

  float acc[4][4] = {};
  for (int tap = 0; tap < taps; ++tap) {
    const int kh = tap / g.Kw, kw = tap - kh * g.Kw;
    const int hn = h + g.ph - kh, wn = w + g.pw - kw;
    bool pix_ok = m_ok && hn >= 0 && wn >= 0 && (hn % g.sh) == 0 && (wn % g.sw) == 0;
    const int ho = hn / g.sh, wo = wn / g.sw;
    pix_ok = pix_ok && ho < g.Ho && wo < g.Wo;
    const long long pix = (long long)ho * g.Wo + wo;
    for (int kb = 0; kb < g.Cot; ++kb) {
      float va[8], vb[8];
      if (pix_ok) {
        const float s = act_scale(a, a.b_scales, tb, pix, n, kb * 32 + kq * 8, g.N, g.Cop);
        decode8<FG>(a.b_codes, (pix * g.N + n) * g.Cop + kb * 32 + kq * 8, s, va, a.fmt_b);
      } else zero8(va);
      const int co = kb * 32 + k_l;
      if (ci_ok && co < g.Cout) {
        const float s = w_scale(a, a.a_scales, ta, co, taps, tap, ci0, g.Cp);
        decode8<FW>(a.a_codes, ((long long)co * taps + tap) * g.Cp + ci0, s, vb, a.fmt_a);
      } else zero8(vb);
      __syncthreads();
      store_kmajor(sm.As, row_l, kq, va);
      store_mnmajor(sm.Bs, k_l, nq, vb);
      __syncthreads();
      mma_tile(sm, ty, tx, acc);
    }
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const long long mm = m0 + ty * 4 + i;
    if (mm >= M) continue;
    const int nn = (int)(mm % g.N); const long long q = mm / g.N;
    const int ww = (int)(q % g.W), hh = (int)(q / g.W);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int c = n0 + tx * 4 + j;
      if (c >= g.Cin) continue;
      if (a.out_layout == MQ_NCHW) a.out[(((long long)nn * g.Cin + c) * g.H + hh) * g.W + ww] = acc[i][j];
      else a.out[mm * g.Cin + c] = acc[i][j];
    }
  }
}

// -------------------------------------------------------------------------------- weight gradient
// Partial sums over a slice of output pixels go to workspace [split][C_out][taps*Cp]; a second
// kernel adds the slices in a fixed order and writes G_W in its final layout.
template <int FX, int FG>
__global__ void __launch_bounds__(GT) bwd_weight_generic(ConvArgs a, int splits) {
  __shared__ Tiles sm;
  const Geom& g = a.g;
  const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15;
  const int k_l = tid >> 3, q8 = tid & 7;
  const int m0 = blockIdx.x * TM, n0 = blockIdx.y * TN;
  const int taps = g.Kh * g.Kw;
  const int J = taps * g.Cp;
  const int npix = g.Ho * g.Wo;
  const int split = blockIdx.z;
  const int pix_begin = (int)((long long)npix * split / splits), pix_end = (int)((long long)npix * (split + 1) / splits);

  const int co0 = m0 + q8 * 8;
  const bool co_ok = co0 < g.Cop;
  const int j0 = n0 + q8 * 8;
  const bool j_ok = j0 < J;
  const int tap = j_ok ? j0 / g.Cp : 0, ci0 = j_ok ? j0 - tap * g.Cp : 0;
  const int kh = tap / g.Kw, kw = tap - kh * g.Kw;
  const float ta = a.ts16 ? *a.a_tscale : 1.f, tb = a.ts16 ? *a.b_tscale : 1.f;

  float acc[4][4] = {};
  for (int pix = pix_begin; pix < pix_end; ++pix) {
    const int ho = pix / g.Wo, wo = pix - ho * g.Wo;
    const int h = ho * g.sh + kh - g.ph, w = wo * g.sw + kw - g.pw;
    const bool x_ok = j_ok && h >= 0 && h < g.H && w >= 0 && w < g.W;
    const long long xpix = (long long)h * g.W + w;
    for (int kb = 0; kb < g.Nt; ++kb) {
      const int n = kb * 32 + k_l;
      float va[8], vb[8];
      if (co_ok && n < g.N) {
        const float s = act_scale(a, a.b_scales, tb, pix, n, co0, g.N, g.Cop);
        decode8<FG>(a.b_codes, ((long long)pix * g.N + n) * g.Cop + co0, s, va, a.fmt_b);
      } else zero8(va);
      if (x_ok && n < g.N) {
        const float s = act_scale(a, a.a_scales, ta, xpix, n, ci0, g.N, g.Cp);
        decode8<FX>(a.a_codes, (xpix * g.N + n) * g.Cp + ci0, s, vb, a.fmt_a);
      } else zero8(vb);
      __syncthreads();
      store_mnmajor(sm.As, k_l, q8, va);
      store_mnmajor(sm.Bs, k_l, q8, vb);
      __syncthreads();
      mma_tile(sm, ty, tx, acc);
    }
  }
  float* part = reinterpret_cast<float*>(a.workspace) + (long long)split * g.Cout * J;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int co = m0 + ty * 4 + i;
    if (co >= g.Cout) continue;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int jj = n0 + tx * 4 + j;
      if (jj < J) part[(long long)co * J + jj] = acc[i][j];
    }
  }
}

// ---- sums of the split-K partials [split][Cout][taps][Cp], added in a fixed order and written in G_W's final layout -----------------
// Reads are 16 bytes per thread, consecutive threads along the partials' own order; `groups` neighbouring thread groups share a
// block's sums (every groups-th split each, combined through shared memory in group order: independent of scheduling).
// ta, tb: the two tensors' fp32 scales when the partial sums still lack them (tensor-core GEMM on E4M3-scaled blocks, Eq. 4), else null
constexpr int RED_THREADS = 256, RED_RUNS_MAX = 512;
template <int GROUPS>
__device__ __forceinline__ float4 sum_of_splits(const float4* p, long long slab4, int grp, int splits) {
  float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
  for (int k = grp; k < splits; k += GROUPS) {
    const float4 v = __ldg(p + (long long)k * slab4);
    s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w;
  }
  return s;
}
// adds the other groups' sums to group 0's (threads of group q hold theirs `per` threads apart)
template <int GROUPS>
__device__ __forceinline__ void sum_of_groups(float4& s, float4* sh, int grp, int per) {
  if (GROUPS == 1) return;
  if (grp > 0 && grp < GROUPS) sh[threadIdx.x] = s;
  __syncthreads();
  if (grp == 0) {
#pragma unroll
    for (int q = 1; q < GROUPS; ++q) { const float4 v = sh[threadIdx.x + q * per]; s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w; }
  }
}
// Any layer: a block takes RED_THREADS / GROUPS consecutive float4s of the partials.
template <int GROUPS>
__global__ void __launch_bounds__(RED_THREADS) bwd_weight_reduce(const float* __restrict__ part, float* __restrict__ out, Geom g, int splits, int layout,
                                                                 const float* __restrict__ ta, const float* __restrict__ tb) {
  pdl_wait();
  __shared__ float4 sh[RED_THREADS];
  constexpr int per = RED_THREADS / GROUPS;
  const float os = ta ? __ldg(ta) * __ldg(tb) : 1.f;
  const int taps = g.Kh * g.Kw;
  const int cq = g.Cp >> 2;                                   // float4 columns per (co, tap)
  const long long quads = (long long)g.Cout * taps * cq;
  const int grp = (int)threadIdx.x / per, col = (int)threadIdx.x % per;
  for (long long base = (long long)blockIdx.x * per; base < quads; base += (long long)gridDim.x * per) {
    const long long qd = base + col;
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
    if (qd < quads) s = sum_of_splits<GROUPS>(reinterpret_cast<const float4*>(part) + qd, quads, grp, splits);
    sum_of_groups<GROUPS>(s, sh, grp, per);
    if (grp == 0 && qd < quads) {
      const int c4 = (int)(qd % cq); const long long r = qd / cq;
      const int tap = (int)(r % taps), co = (int)(r / taps), ci0 = 4 * c4;
      const float vals[4] = {s.x * os, s.y * os, s.z * os, s.w * os};
      const bool rows = layout != MQ_NCHW || taps == 1;       // channel-fastest
      float* o = rows ? out + ((long long)co * taps + tap) * g.Cin + ci0 : out + ((long long)co * g.Cin + ci0) * taps + tap;
      if (rows && (g.Cin & 3) == 0) { if (ci0 < g.Cin) *reinterpret_cast<float4*>(o) = make_float4(vals[0], vals[1], vals[2], vals[3]); }
      else {
#pragma unroll
        for (int e = 0; e < 4; ++e) if (ci0 + e < g.Cin) o[(long long)e * (rows ? 1 : taps)] = vals[e];
      }
    }
    __syncthreads();
  }
}
// [C_out][C_in][taps] results of layers with many channels.  There the four channels that a thread has added lie taps floats apart, a
// sector each, and those stores take longer than the reads; so a block takes all taps of R channels of one output channel, which
// G_W holds as one run, turns them in shared memory and stores whole lines.  (Whole call, before -> now: 512 -> 512 channels 14x14, E2M1,
// N = 256, 3 splits 85.5 -> 75.7 us, N = 64 41.8 -> 31.8; 256 -> 256 14x14, N = 64, 12 splits 22.1 -> 19.4.)
template <int GROUPS>
__global__ void __launch_bounds__(RED_RUNS_MAX) bwd_weight_reduce_runs(const float* __restrict__ part, float* __restrict__ out, Geom g, int splits, int R, int nr,
                                                                       int per, const float* __restrict__ ta, const float* __restrict__ tb) {
  pdl_wait();
  extern __shared__ __align__(16) float red_stage[];          // [R][taps]
  __shared__ float4 sh[RED_RUNS_MAX];
  const float os = ta ? __ldg(ta) * __ldg(tb) : 1.f;
  const int taps = g.Kh * g.Kw;
  const long long slab4 = (long long)g.Cout * taps * (g.Cp >> 2);     // float4s per split
  const int co = (int)blockIdx.x / nr, ci0 = ((int)blockIdx.x - co * nr) * R;
  const int rq = min(R, g.Cp - ci0) >> 2, nq = taps * rq;
  const int grp = (int)threadIdx.x / per, i = (int)threadIdx.x - grp * per;
  const int tap = i / rq, c = 4 * (i - tap * rq);
  float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
  if (grp < GROUPS && i < nq)      // (the block's last warp may be only partly in use)
    s = sum_of_splits<GROUPS>(reinterpret_cast<const float4*>(part + ((long long)co * taps + tap) * g.Cp + ci0 + c), slab4, grp, splits);
  sum_of_groups<GROUPS>(s, sh, grp, per);
  if (grp == 0 && i < nq) {
    red_stage[c * taps + tap] = s.x * os; red_stage[(c + 1) * taps + tap] = s.y * os;
    red_stage[(c + 2) * taps + tap] = s.z * os; red_stage[(c + 3) * taps + tap] = s.w * os;
  }
  __syncthreads();
  const int n = min(R, g.Cin - ci0) * taps;       // (channels of the padding are left out)
  float* o = out + ((long long)co * g.Cin + ci0) * taps;
  for (int k = threadIdx.x; k < n; k += blockDim.x) o[k] = red_stage[k];
}

}  // namespace

int conv_generic_bwd_weight_splits(const Geom& g) {
  const int taps = g.Kh * g.Kw;
  const long long tiles = (long long)((g.Cop + TM - 1) / TM) * ((taps * g.Cp + TN - 1) / TN);
  long long splits = ((long long)sm_count() * 4 + tiles - 1) / tiles;
  const long long npix = (long long)g.Ho * g.Wo;
  if (splits > npix) splits = npix;
  if (splits > 256) splits = 256;
  if (splits < 1) splits = 1;
  return (int)splits;
}

size_t conv_generic_workspace(int op, const Geom& g) {
  if (op != MQ_OP_BWD_WEIGHT) return 0;
  return (size_t)conv_generic_bwd_weight_splits(g) * g.Cout * g.Kh * g.Kw * g.Cp * sizeof(float);
}

cudaError_t launch_bwd_weight_reduce(const float* partial, float* out, const Geom& g, int splits, int layout, cudaStream_t s, const float* ta,
                                     const float* tb) {
  const int taps = g.Kh * g.Kw, sms = sm_count();
  count_launches(1);
  // Whole runs: blocks of 64 or 128 channels (two lines per read, at least) that give every SM two, and more with many splits, where the
  // reads are what takes the time and the other kernel has more threads in flight (whole call, 96 -> 160 channels 27x27, 320 blocks, 24
  // splits: 24.1 us as runs, 22.1; 64 -> 320 102x178 stride 2, 320, 16: 28.9 / 27.3; 256 -> 256 28x28, 512, 12: 87.6 / 91.8).
  for (int R = 128; R >= 64 && layout == MQ_NCHW && taps > 1; R /= 2) {
    const int nr = (g.Cp + R - 1) / R, per = taps * (R / 4);
    const long long units = (long long)g.Cout * nr;
    if (R > g.Cp || per > RED_RUNS_MAX || 4 * units < sms * (splits > 8 ? splits : 8) || units > 0x7fffffffLL) continue;
    const bool two = 2 * per <= RED_RUNS_MAX && splits > 1;
    const unsigned threads = (unsigned)((two ? 2 : 1) * per + 31) / 32 * 32;
    return launch_pdl(two ? bwd_weight_reduce_runs<2> : bwd_weight_reduce_runs<1>, dim3((unsigned)units), dim3(threads), (size_t)R * taps * sizeof(float), s,
                      partial, out, g, splits, R, nr, per, ta, tb);
  }
  // four groups, more where that leaves SMs idle and a group still has a few splits to add (32 -> 32 channels 32x32, 49 splits, the call:
  // 9.9 us with four, 9.1 with sixteen)
  const long long quads = (long long)g.Cout * taps * (g.Cp / 4);
  int groups = 4;
  while (groups < 16 && quads * groups < 512ll * sms && splits >= 4 * groups) groups *= 2;
  const int per = RED_THREADS / groups;
  unsigned blocks = (unsigned)((quads + per - 1) / per);
  if (blocks > (unsigned)sms * 16) blocks = (unsigned)sms * 16;
  auto kernel = groups == 4 ? bwd_weight_reduce<4> : groups == 8 ? bwd_weight_reduce<8> : bwd_weight_reduce<16>;
  return launch_pdl(kernel, dim3(blocks), dim3(RED_THREADS), 0, s, partial, out, g, splits, layout, ta, tb);
}

// Two template classes per operand: packed E2M1 (2) or one byte per code (0; the format itself is read at run time)
#define MQ_DISPATCH2(FA, FB, CALL)                                                         \
  switch (((FA) == MQ_E2M1 ? 2 : 0) + ((FB) == MQ_E2M1 ? 1 : 0)) {                            \
    case 0: { constexpr int A_ = 0, B_ = 0; CALL; } break;                                 \
    case 1: { constexpr int A_ = 0, B_ = 2; CALL; } break;                                 \
    case 2: { constexpr int A_ = 2, B_ = 0; CALL; } break;                                 \
    case 3: { constexpr int A_ = 2, B_ = 2; CALL; } break;                                 \
    default: return cudaErrorInvalidValue;                                                 \
  }

cudaError_t launch_conv_generic(int op, const ConvArgs& a, cudaStream_t s) {
  const Geom& g = a.g;
  if (op == MQ_OP_FWD) {
    const long long M = (long long)g.Ho * g.Wo * g.N;
    dim3 grid((unsigned)((M + TM - 1) / TM), (unsigned)((g.Cout + TN - 1) / TN));
    MQ_DISPATCH2(a.fmt_a, a.fmt_b, (fwd_generic<A_, B_><<<grid, GT, 0, s>>>(a)));
  } else if (op == MQ_OP_BWD_DATA) {
    const long long M = (long long)g.H * g.W * g.N;
    dim3 grid((unsigned)((M + TM - 1) / TM), (unsigned)((g.Cin + TN - 1) / TN));
    MQ_DISPATCH2(a.fmt_a, a.fmt_b, (bwd_data_generic<A_, B_><<<grid, GT, 0, s>>>(a)));
  } else {
    const int splits = conv_generic_bwd_weight_splits(g);
    const int J = g.Kh * g.Kw * g.Cp;
    dim3 grid((unsigned)((g.Cop + TM - 1) / TM), (unsigned)((J + TN - 1) / TN), (unsigned)splits);
    MQ_DISPATCH2(a.fmt_a, a.fmt_b, (bwd_weight_generic<A_, B_><<<grid, GT, 0, s>>>(a, splits)));
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    e = launch_bwd_weight_reduce(reinterpret_cast<const float*>(a.workspace), a.out, g, splits, a.out_layout, s, nullptr, nullptr);
    if (e != cudaSuccess) return e;
  }
  count_launches(1);
  return cudaGetLastError();
}

}  // namespace mq
