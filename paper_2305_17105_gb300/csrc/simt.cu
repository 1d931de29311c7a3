// FP32 CUDA-core form of the NTC hot path: random-access decode (nearest,
// trilinear, stochastic) and the fused forward + loss + backward of the
// optimisation (Sec. 4.3-4.5, 5.1, 5.3).  The MLP runs as register-tiled
// FP32 matrix products on tiles of 32 queries / texels whose activations stay
// in shared memory; every activation is recomputed on chip.
#include <cooperative_groups.h>

#include "ntc_device.cuh"
#include "ntc_internal.h"

namespace ntc {

namespace {

// ---------------------------------------------------------------------------
// Decode.  A warp owns a tile of 32 queries.  Its input rows (and, in place,
// the hidden rows) lie in shared memory unit-major, act[unit][kLd] with the
// 32 queries contiguous, and lane (qg = lane / 8, ng = lane % 8) computes the
// outputs n = ng + 8 j of queries 4 qg .. +3 and 16 + 4 qg .. +3: 64 FP32
// accumulators for a 64-wide layer, four 16-byte shared loads per 64 FMAs.
// The FMA chain of every output runs over k in order from the bias, so the
// values are those of a plain loop.  kLd = 36 puts eight consecutive units
// on disjoint banks for the 16-byte stores of a quarter-warp.
// What bounds it: the FP32 FMA rate (78.4 TFLOP/s measured).  One thread per
// query with every weight broadcast from shared memory (the form this
// replaced) needed a 16-byte load per four FMAs and was bound by them:
// a pass of 65,536 queries of a 256^2 x 8 material took 86 us against 29 now
// (22 of them the host's share of a call).
// ---------------------------------------------------------------------------
constexpr int kLd = 36;         // floats per unit row: 32 queries + 4 of padding
constexpr int kMaxWarps = 16;   // tiles in flight per CTA (one CTA per SM)

// Shared-memory weights of the decode, in floats: hidden layers [k][64] with
// output n = ng + 8 j at 32 (j / 4) + 4 ng + j % 4, the output layer [64][16]
// with n = ng + 8 j at 2 ng + j (rows >= C zero), biases, then one activation
// region per warp (`rows` units and the 32 blend weights of trilinear taps).
struct SW {
  int w1, w2, w3, b1, b2, b3, wh, bh, act, warp;
  bool h3;
  __host__ __device__ SW(int K, bool third) {
    w1 = 0;
    w2 = w1 + K * kHidden;
    w3 = w2 + kHidden * kHidden;
    b1 = w3 + kMaxC * kHidden;
    b2 = b1 + kHidden;
    b3 = b2 + kHidden;
    wh = b3 + kMaxC;
    bh = wh + (third ? kHidden * kHidden : 0);
    act = bh + (third ? kHidden : 0);
    warp = (K > kHidden ? K : kHidden) * kLd + 32;
    h3 = third;
  }
  __host__ __device__ size_t bytes(int warps) const { return (size_t)(act + warps * warp) * 4; }
};

// Four consecutive inputs k .. k + 3 (k a multiple of 4) of row o of a
// weight matrix [rows][ld] in the material's precision.
__device__ __forceinline__ float4 weight4(const ntc_material& M, const void* w, float scale, int i) {
  switch (M.precision) {
    case NTC_PREC_F16: {
      const uint2 v = __ldg(reinterpret_cast<const uint2*>(static_cast<const __half*>(w) + i));
      union { uint32_t u; __half2 h; } a, b;
      a.u = v.x;
      b.u = v.y;
      const float2 lo = __half22float2(a.h), hi = __half22float2(b.h);
      return make_float4(lo.x, lo.y, hi.x, hi.y);
    }
    case NTC_PREC_F8: {
      const __nv_fp8_e4m3* e = static_cast<const __nv_fp8_e4m3*>(w) + i;
      return make_float4((float)e[0] * scale, (float)e[1] * scale, (float)e[2] * scale,
                         (float)e[3] * scale);
    }
    default: return __ldg(reinterpret_cast<const float4*>(static_cast<const float*>(w) + i));
  }
}

// Stage W [64][ld] so that place(o) + 64 k holds (o, k): lanes take
// consecutive outputs, which `place` puts on different banks.
template <class Place>
__device__ __forceinline__ void stage_hidden(const ntc_material& M, const void* w, float scale,
                                             int ld, float* dst, Place place) {
#pragma unroll 4
  for (int i = threadIdx.x; i < kHidden * (ld / 4); i += blockDim.x) {
    const int o = i & (kHidden - 1), k = 4 * (i >> 6);
    const float4 v = weight4(M, w, scale, o * ld + k);
    float* d = dst + place(o) + k * kHidden;
    d[0] = v.x;
    d[kHidden] = v.y;
    d[2 * kHidden] = v.z;
    d[3 * kHidden] = v.w;
  }
}

__device__ void stage_weights(const ntc_material& M, const SW& L, float* s) {
  const int C = M.channels, K = M.k_in;
  const bool f8 = M.precision == NTC_PREC_F8;
  auto place = [](int o) { return 32 * (o >> 5) + 4 * (o & 7) + ((o >> 3) & 3); };
  stage_hidden(M, M.w[0], f8 ? M.scale[0] : 1.f, K, s + L.w1, place);
  stage_hidden(M, M.w[1], f8 ? M.scale[1] : 1.f, kHidden, s + L.w2, place);
  for (int i = threadIdx.x; i < kMaxC * (kHidden / 4); i += blockDim.x) {
    const int c = i & (kMaxC - 1), k = 4 * (i >> 4);
    const float4 v = c < C ? weight4(M, M.w[2], f8 ? M.scale[2] : 1.f, c * kHidden + k)
                           : make_float4(0.f, 0.f, 0.f, 0.f);
    float* d = s + L.w3 + 2 * (c & 7) + (c >> 3) + k * kMaxC;
    d[0] = v.x;
    d[kMaxC] = v.y;
    d[2 * kMaxC] = v.z;
    d[3 * kMaxC] = v.w;
  }
  for (int i = threadIdx.x; i < kHidden; i += blockDim.x) {
    s[L.b1 + i] = M.b[0][i];
    s[L.b2 + i] = M.b[1][i];
    if (L.h3) s[L.bh + i] = M.b_h3[i];
  }
  for (int i = threadIdx.x; i < kMaxC; i += blockDim.x) s[L.b3 + i] = i < C ? M.b[2][i] : 0.f;
  if (L.h3) stage_hidden(M, M.w_h3, 1.f, kHidden, s + L.wh, place);
}

// The lane's J outputs n = ng + 8 j (J = 8: a hidden layer, J = 2: the output
// layer) of its eight queries: z[j][p] holds queries 4 qg + {0,1}, {2,3} and
// 16 + 4 qg + {0,1}, {2,3}.
template <int J>
__device__ __forceinline__ void warp_dense(const float* __restrict__ W, const float* __restrict__ b,
                                           const float* __restrict__ act, int K, int lane,
                                           float2 (&z)[J][4]) {
  const int ng = lane & 7, qg = lane >> 3;
#pragma unroll
  for (int j = 0; j < J; ++j) {
    const float bj = b[ng + 8 * j];
#pragma unroll
    for (int p = 0; p < 4; ++p) z[j][p] = make_float2(bj, bj);
  }
  const float* xp = act + 4 * qg;
  const float* wp = W + (J == 8 ? 4 : 2) * ng;
#pragma unroll 4
  for (int k = 0; k < K; ++k) {
    const float4 xa = *reinterpret_cast<const float4*>(xp + k * kLd);
    const float4 xb = *reinterpret_cast<const float4*>(xp + k * kLd + 16);
    float w[J];
    if constexpr (J == 8) {
      const float4 w0 = *reinterpret_cast<const float4*>(wp + k * kHidden);
      const float4 w1 = *reinterpret_cast<const float4*>(wp + k * kHidden + 32);
      w[0] = w0.x; w[1] = w0.y; w[2] = w0.z; w[3] = w0.w;
      w[4] = w1.x; w[5] = w1.y; w[6] = w1.z; w[7] = w1.w;
    } else {
      const float2 w0 = *reinterpret_cast<const float2*>(wp + k * kMaxC);
      w[0] = w0.x; w[1] = w0.y;
    }
#pragma unroll
    for (int j = 0; j < J; ++j) {
      const float2 ww = make_float2(w[j], w[j]);
      z[j][0] = __ffma2_rn(ww, make_float2(xa.x, xa.y), z[j][0]);
      z[j][1] = __ffma2_rn(ww, make_float2(xa.z, xa.w), z[j][1]);
      z[j][2] = __ffma2_rn(ww, make_float2(xb.x, xb.y), z[j][2]);
      z[j][3] = __ffma2_rn(ww, make_float2(xb.z, xb.w), z[j][3]);
    }
  }
}

// act(z) of a hidden layer -> the warp's unit rows, once every lane has read
// the layer's input.
__device__ __forceinline__ void put_hidden(float* act, int lane, int fn, float2 (&z)[8][4]) {
  __syncwarp();
  float* p = act + (lane & 7) * kLd + 4 * (lane >> 3);
  auto apply = [&](int f) {
#pragma unroll
    for (int j = 0; j < 8; ++j)
#pragma unroll
      for (int i = 0; i < 4; ++i) z[j][i] = make_float2(act_fwd(f, z[j][i].x), act_fwd(f, z[j][i].y));
  };
  if (fn == NTC_ACT_RELU) apply(NTC_ACT_RELU);
  else apply(NTC_ACT_HARDGELU);
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    *reinterpret_cast<float4*>(p + 8 * j * kLd) = make_float4(z[j][0].x, z[j][0].y, z[j][1].x, z[j][1].y);
    *reinterpret_cast<float4*>(p + 8 * j * kLd + 16) = make_float4(z[j][2].x, z[j][2].y, z[j][3].x, z[j][3].y);
  }
  __syncwarp();
}

// Input rows are written one query per lane: unit i of this lane's column.
struct ColumnSink {
  float* col;
  __device__ __forceinline__ void operator()(int i, float v) const { col[i * kLd] = v; }
};

// One output element of the decode.
__device__ __forceinline__ void store_value(void* out, int out_dtype, int64_t e, float y) {
  if (out_dtype == NTC_DTYPE_F32) static_cast<float*>(out)[e] = y;
  else if (out_dtype == NTC_DTYPE_U8)
    static_cast<uint8_t*>(out)[e] = (uint8_t)__float2uint_rn(__saturatef(y) * 255.f);
  else static_cast<__half*>(out)[e] = __float2half_rn(y);
}

__global__ void __launch_bounds__(32 * kMaxWarps, 1) decode_simt_kernel(
    const ntc_material M, const float* __restrict__ uvl, int64_t n, void* __restrict__ out,
    int out_dtype, int filter, int noise, uint64_t nkey, uint64_t jkey) {
  extern __shared__ __align__(16) float smem[];
  const int K = M.k_in, C = M.channels;
  const SW L(K, M.hidden_layers == 3);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
  stage_weights(M, L, smem);
  __syncthreads();
  float* act = smem + L.act + warp * L.warp;
  float* wtap = act + L.warp - 32;
  ColumnSink sink{act + lane};
  const int ng = lane & 7, qg = lane >> 3;
  const bool tri = filter == NTC_FILTER_TRILINEAR;
  const int64_t tiles = (n + 31) / 32;
  for (int64_t t = blockIdx.x + (int64_t)warp * gridDim.x; t < tiles; t += (int64_t)gridDim.x * warps) {
    // the lanes past the last query repeat it; their outputs are not stored
    const int64_t q = min(t * 32 + lane, n - 1);
    const float u = uvl[3 * q], v = uvl[3 * q + 1], l = uvl[3 * q + 2];
    float2 y[2][4];
#pragma unroll 1
    for (int tap = 0; tap < (tri ? 8 : 1); ++tap) {
      int x, yy, m;
      if (filter == NTC_FILTER_NEAREST) {
        query_texel(M, u, v, l, x, yy, m);
      } else if (filter == NTC_FILTER_STOCHASTIC) {
        const uint64_t h = splitmix64(jkey ^ (uint64_t)q);
        m = stochastic_mip(l, M.mips, h);
        x = stochastic_coord(u, mip_dim(M.width, m), (uint32_t)(h >> 40));
        yy = stochastic_coord(v, mip_dim(M.height, m), (uint32_t)(h >> 16) & 0xFFFFFFu);
      } else {
        // software trilinear filtering (Sec. 5.3): 2x2 texels on two mips
        const float lam = !(l >= 0.f) ? 0.f : fminf(l, (float)(M.mips - 1));
        const int m0 = min((int)floorf(lam), M.mips - 1);
        const int m1 = min(m0 + 1, M.mips - 1);
        const float tl = lam - (float)m0;
        const int s = tap >> 2, dx = tap & 1, dy = (tap >> 1) & 1;
        m = s ? m1 : m0;
        const float wl = s ? tl : 1.f - tl;
        const int wm = mip_dim(M.width, m), hm = mip_dim(M.height, m);
        const float px = u * (float)wm - 0.5f, py = v * (float)hm - 0.5f;
        const float fx0 = floorf(px), fy0 = floorf(py);
        const float fx = px - fx0, fy = py - fy0;
        x = wrap_texel((int)fx0 + dx, wm);
        yy = wrap_texel((int)fy0 + dy, hm);
        wtap[lane] = wl * (dx ? fx : 1.f - fx) * (dy ? fy : 1.f - fy);
      }
      featurize(M, x, yy, m, noise != 0, nkey, sink);
      __syncwarp();
      // the hidden layers (two, or three: Sec. 4.4), one body
#pragma unroll 1
      for (int l = 0; l < (L.h3 ? 3 : 2); ++l) {
        const float* w = smem + (l == 0 ? L.w1 : (l == 1 ? L.w2 : L.wh));
        const float* b = smem + (l == 0 ? L.b1 : (l == 1 ? L.b2 : L.bh));
        float2 z[8][4];
        warp_dense<8>(w, b, act, l == 0 ? K : kHidden, lane, z);
        put_hidden(act, lane, M.act, z);
      }
      float2 o[2][4];
      warp_dense<2>(smem + L.w3, smem + L.b3, act, kHidden, lane, o);
#pragma unroll
      for (int j = 0; j < 2; ++j)
#pragma unroll
        for (int p = 0; p < 4; ++p) {
          const float2 yo = make_float2(out_fwd(M.out_act, o[j][p].x), out_fwd(M.out_act, o[j][p].y));
          if (!tri) {
            y[j][p] = yo;
          } else {
            const float2 w = *reinterpret_cast<const float2*>(wtap + 16 * (p >> 1) + 4 * qg + 2 * (p & 1));
            const float2 y0 = tap ? y[j][p] : make_float2(0.f, 0.f);
            y[j][p] = make_float2(fmaf(w.x, yo.x, y0.x), fmaf(w.y, yo.y, y0.y));
          }
        }
      __syncwarp();  // the next tile's rows overwrite the activations
    }
#pragma unroll
    for (int p = 0; p < 4; ++p)
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const int64_t qo = t * 32 + 16 * (p >> 1) + 4 * qg + 2 * (p & 1) + e;
        if (qo < n) {
          if (ng < C) store_value(out, out_dtype, qo * C + ng, e ? y[0][p].y : y[0][p].x);
          if (ng + 8 < C) store_value(out, out_dtype, qo * C + ng + 8, e ? y[1][p].y : y[1][p].x);
        }
      }
  }
}

// Calibration of the FP8-E4M3 form: the largest magnitude of each layer's
// input (the feature row, act(Z1), act(Z2)) over the nearest decodes of the
// queries, in FP32, reduced per warp and merged into amax[3] (float bits;
// every value is non-negative, so the unsigned order is the float order).
__global__ void __launch_bounds__(32 * kMaxWarps, 1) f8_calib_kernel(const ntc_material M,
                                                                     const float* __restrict__ uvl,
                                                                     int64_t n, uint32_t* amax) {
  extern __shared__ __align__(16) float smem[];
  const int K = M.k_in;
  const SW L(K, false);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
  stage_weights(M, L, smem);
  __syncthreads();
  float* act = smem + L.act + warp * L.warp;
  ColumnSink sink{act + lane};
  float mx[3] = {0.f, 0.f, 0.f};
  auto merge = [](float& a, const float2 (&z)[8][4]) {
#pragma unroll
    for (int j = 0; j < 8; ++j)
#pragma unroll
      for (int p = 0; p < 4; ++p) a = fmaxf(a, fmaxf(fabsf(z[j][p].x), fabsf(z[j][p].y)));
  };
  const int64_t tiles = (n + 31) / 32;
  for (int64_t t = blockIdx.x + (int64_t)warp * gridDim.x; t < tiles; t += (int64_t)gridDim.x * warps) {
    const int64_t q = min(t * 32 + lane, n - 1);  // the last query again past the end
    int x, yy, m;
    query_texel(M, uvl[3 * q], uvl[3 * q + 1], uvl[3 * q + 2], x, yy, m);
    featurize(M, x, yy, m, false, 0, sink);
    for (int k = 0; k < K; ++k) mx[0] = fmaxf(mx[0], fabsf(sink.col[k * kLd]));
    __syncwarp();
    float2 z[8][4];
    warp_dense<8>(smem + L.w1, smem + L.b1, act, K, lane, z);
    put_hidden(act, lane, M.act, z);
    merge(mx[1], z);
    warp_dense<8>(smem + L.w2, smem + L.b2, act, kHidden, lane, z);
    put_hidden(act, lane, M.act, z);
    merge(mx[2], z);
  }
#pragma unroll
  for (int l = 0; l < 3; ++l) {
    float v = mx[l];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    if (lane == 0) atomicMax(&amax[l], __float_as_uint(v));
  }
}

// amax[3] (float bits) -> the activation scales s_a[l]: the smallest power
// of two with amax / s_a <= 448 (the largest finite E4M3 value); 1 for an
// all-zero input.
__global__ void f8_scales_kernel(const uint32_t* amax, float* sa) {
  const int l = threadIdx.x;
  if (l >= 3) return;
  const float a = __uint_as_float(amax[l]);
  float s = 1.f;
  if (a > 0.f && a < __int_as_float(0x7f800000)) {
    int e = 0;
    const float f = frexpf(a / 448.f, &e);  // a / 448 = f 2^e, f in [0.5, 1)
    if (f == 0.5f) e -= 1;                    // an exact power of two needs no headroom
    e = e < -126 ? -126 : (e > 127 ? 127 : e);
    s = __int_as_float((127 + e) << 23);
  }
  sa[l] = s;
}

// ---------------------------------------------------------------------------
// Fused forward + loss + backward (Sec. 5.1).  A CTA of 128 threads takes
// tiles of 32 texels; units lie unit-major in shared memory as in the decode,
// and thread (qg, ng) computes outputs n = ng + 16 j (j < 4) of texels 4 qg ..
// +3 of every product (16 accumulators).  Per tile:
//   features -> X;  Z1, H1 = act(Z1);  Z2, H2;  Z3 -> loss, D3;
//   dW3 += D3 H2^T, D2 = (W3^T D3) act'(Z2) over H2;
//   dW2 += D2 H1^T, D1 = (W2^T D2) act'(Z1) over H1;
//   dW1 += D1 X^T,  dX = W1^T D1 -> scatter-add through the taps.
// act' stays in the registers of the thread that owns the unit; the weight
// gradients stay in registers over all tiles of the CTA (72 per thread: 4x8
// blocks of dW1 and dW2, 1x8 of dW3) and leave once, staged row-major, as
// vector reductions.
// What bounds it: for a batch of a few thousand texels the serial chain of
// one tile, hence small tiles spread over all SMs, with the rows' features
// split over the warps (G0, G1, the encoding and target, the taps).  Tiles
// of 128 texels, one per thread, ran a 4,096-texel step of a 256^2 x 8
// material on 32 CTAs in 118 us (all launches of the step) against 37 now.
// ---------------------------------------------------------------------------
constexpr int kBTile = 32;
constexpr int kBThreads = 128;
constexpr int kBCluster = 4;   // CTAs that add their losses before one of them reduces
constexpr int kTapMeta = 112;  // bytes per texel: 8 cell addresses, 8 weights, padding

struct SB {
  int w1f, w2f, w3f, w1b, w2b, w3b, b1, b2, b3, x, h1, h2, d3, meta, red, size;
  __host__ __device__ explicit SB(int K) {
    w1f = 0;                               // [K][64], output n = ng + 16 j at 4 ng + j
    w2f = w1f + K * kHidden;               // [64][64]
    w3f = w2f + kHidden * kHidden;         // [64][16]
    w1b = w3f + kMaxC * kHidden;           // transposed for the backward: [64 o][64 slots]
    w2b = w1b + kHidden * kHidden;         // [64 o][64 i]
    w3b = w2b + kHidden * kHidden;         // [16 c][64 i]
    b1 = w3b + kMaxC * kHidden;
    b2 = b1 + kHidden;
    b3 = b2 + kHidden;
    x = b3 + kMaxC;                        // unit-major tiles, kLd floats per unit
    h1 = x + K * kLd;
    h2 = h1 + kHidden * kLd;
    d3 = h2 + kHidden * kLd;
    meta = d3 + kMaxC * kLd;
    red = meta + kBTile * kTapMeta / 4;    // [4]
    size = red + 4;
  }
};

__device__ __forceinline__ int place16(int n) { return 4 * (n & 15) + (n >> 4); }

// The backward's operand of a hidden layer, [64 o][64] with column k at
// place16(k) (zero from `cols` on), from the forward's [k][64] with output o
// at place16(o).  Lane l of step d moves (o, k) = (l, (l + d) mod 32) of a
// 32 x 32 block, so both sides hit 32 different banks.
__device__ __forceinline__ void transpose_hidden(const float* __restrict__ f, int cols,
                                                 float* __restrict__ dst) {
  const int l = threadIdx.x & 31;
#pragma unroll 4
  for (int i = threadIdx.x >> 5; i < 4 * 32; i += kBThreads / 32) {
    const int o = 32 * (i >> 6) + l, k = 32 * ((i >> 5) & 1) + ((l + i) & 31);
    dst[o * kHidden + place16(k)] = k < cols ? f[k * kHidden + place16(o)] : 0.f;
  }
}

// z[j] += the thread's outputs ng + 16 j of its four texels, over `rows`
// units of `in` ([unit][kLd]) against W [unit][64].
__device__ __forceinline__ void tile_dense(const float* __restrict__ W, const float* __restrict__ in,
                                           int rows, int ng, int qg, float2 (&z)[4][2]) {
  const float* xp = in + 4 * qg;
  const float* wp = W + 4 * ng;
#pragma unroll 4
  for (int k = 0; k < rows; ++k) {
    const float4 x = *reinterpret_cast<const float4*>(xp + k * kLd);
    const float4 w4 = *reinterpret_cast<const float4*>(wp + k * kHidden);
    const float w[4] = {w4.x, w4.y, w4.z, w4.w};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float2 ww = make_float2(w[j], w[j]);
      z[j][0] = __ffma2_rn(ww, make_float2(x.x, x.y), z[j][0]);
      z[j][1] = __ffma2_rn(ww, make_float2(x.z, x.w), z[j][1]);
    }
  }
}
__device__ __forceinline__ void put_units(float* dst, int ng, int qg, const float2 (&z)[4][2]) {
#pragma unroll
  for (int j = 0; j < 4; ++j)
    *reinterpret_cast<float4*>(dst + (ng + 16 * j) * kLd + 4 * qg) =
        make_float4(z[j][0].x, z[j][0].y, z[j][1].x, z[j][1].y);
}
// z -> act(z), keeping act'(z).
__device__ __forceinline__ void activate(int fn, float2 (&z)[4][2], float2 (&g)[4][2]) {
  auto apply = [&](int f) {
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int p = 0; p < 2; ++p) {
        g[j][p] = make_float2(act_grad(f, z[j][p].x), act_grad(f, z[j][p].y));
        z[j][p] = make_float2(act_fwd(f, z[j][p].x), act_fwd(f, z[j][p].y));
      }
  };
  if (fn == NTC_ACT_RELU) apply(NTC_ACT_RELU);
  else apply(NTC_ACT_HARDGELU);
}

// acc[r][s] += sum over the 32 texels of d[og + 16 r] h[ig + 8 s] (rows of
// units; s < cols / 8).  The tile is summed by itself first: one chain over
// all of a CTA's texels would round every product to the running total
// (2^18 texels, K = 32: 2.8e-7 from 64 bits in dW1).
template <int R>
__device__ __forceinline__ void outer_acc(const float* __restrict__ d, const float* __restrict__ h,
                                          int og, int ig, int cols, float (&acc)[R][8]) {
  float t[R][8] = {};
#pragma unroll 1
  for (int q = 0; q < kBTile; q += 4) {
    float4 dv[R];
#pragma unroll
    for (int r = 0; r < R; ++r) dv[r] = *reinterpret_cast<const float4*>(d + (og + 16 * r) * kLd + q);
#pragma unroll
    for (int s = 0; s < 8; ++s)
      if (8 * s < cols) {
        const float4 hv = *reinterpret_cast<const float4*>(h + (ig + 8 * s) * kLd + q);
#pragma unroll
        for (int r = 0; r < R; ++r) {
          t[r][s] = fmaf(dv[r].x, hv.x, t[r][s]);
          t[r][s] = fmaf(dv[r].y, hv.y, t[r][s]);
          t[r][s] = fmaf(dv[r].z, hv.z, t[r][s]);
          t[r][s] = fmaf(dv[r].w, hv.w, t[r][s]);
        }
      }
  }
#pragma unroll
  for (int r = 0; r < R; ++r)
#pragma unroll
    for (int s = 0; s < 8; ++s) acc[r][s] += t[r][s];
}
__device__ __forceinline__ float row_sum(const float* __restrict__ d) {
  float s = 0.f;
#pragma unroll
  for (int q = 0; q < kBTile; q += 4) {
    const float4 v = *reinterpret_cast<const float4*>(d + q);
    s += (v.x + v.y) + (v.z + v.w);
  }
  return s;
}

// The staged row-major array `src` (n floats, a multiple of 4) times `gs`
// into the gradient at `g`.  With a `mate` (the same array of the other CTA of
// a cluster of two) the sum of the two, each CTA every other block of the
// elements.
__device__ __forceinline__ void flush_rows(float* g, const float* src, const float* mate, int half,
                                           int n, float gs) {
  if (!g) return;
  const int first = threadIdx.x + (mate ? kBThreads * half : 0), step = mate ? 2 * kBThreads : kBThreads;
  if ((reinterpret_cast<uintptr_t>(g) & 15) == 0 && (n & 3) == 0) {
#pragma unroll 4
    for (int i = first; i < n / 4; i += step) {
      float4 v = reinterpret_cast<const float4*>(src)[i];
      if (mate) {
        const float4 o = reinterpret_cast<const float4*>(mate)[i];
        v = make_float4(v.x + o.x, v.y + o.y, v.z + o.z, v.w + o.w);
      }
      atomicAdd(reinterpret_cast<float4*>(g) + i, make_float4(v.x * gs, v.y * gs, v.z * gs, v.w * gs));
    }
  } else {
    for (int i = first; i < n; i += step) atomicAdd(g + i, (mate ? src[i] + mate[i] : src[i]) * gs);
  }
}

__global__ void __launch_bounds__(kBThreads, 2) backward_simt_kernel(const ntc_material M,
                                                                     const BwdArgs A) {
  extern __shared__ __align__(16) float smem[];
  const int K = M.k_in, C = M.channels;
  const bool learned0 = M.interp0 == NTC_INTERP_LEARNED;
  const int W0 = learned0 ? 4 * M.c0 : M.c0;  // width of the G0 slots
  const SB S(K);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int ng = (lane & 7) + 8 * (warp & 1), qg = (lane >> 3) + 4 * (warp >> 1);
  const int ig = lane & 7, og = (lane >> 3) + 4 * warp;
  {
    const bool f8 = M.precision == NTC_PREC_F8;
    const float s1 = f8 ? M.scale[0] : 1.f, s2 = f8 ? M.scale[1] : 1.f, s3 = f8 ? M.scale[2] : 1.f;
    stage_hidden(M, M.w[0], s1, K, smem + S.w1f, place16);
    stage_hidden(M, M.w[1], s2, kHidden, smem + S.w2f, place16);
    for (int i = tid; i < kMaxC * (kHidden / 4); i += kBThreads) {
      const int c = i & (kMaxC - 1), k = 4 * (i >> 4);
      const float4 v = c < C ? weight4(M, M.w[2], s3, c * kHidden + k) : make_float4(0.f, 0.f, 0.f, 0.f);
      float* d = smem + S.w3f + c + k * kMaxC;
      d[0] = v.x;
      d[kMaxC] = v.y;
      d[2 * kMaxC] = v.z;
      d[3 * kMaxC] = v.w;
    }
    for (int i = tid; i < kHidden; i += kBThreads) {
      smem[S.b1 + i] = M.b[0][i];
      smem[S.b2 + i] = M.b[1][i];
    }
    if (tid < kMaxC) smem[S.b3 + tid] = tid < C ? M.b[2][tid] : 0.f;
    __syncthreads();
    transpose_hidden(smem + S.w1f, K, smem + S.w1b);
    transpose_hidden(smem + S.w2f, kHidden, smem + S.w2b);
#pragma unroll 4
    for (int i = tid; i < kMaxC * kHidden; i += kBThreads)
      smem[S.w3b + (i >> 6) * kHidden + place16(i & 63)] = smem[S.w3f + (i & 63) * kMaxC + (i >> 6)];
  }
  const int64_t step = A.step_dev ? *A.step_dev : A.noise_step;
  const uint64_t nkey = rng_key(A.noise_seed, noise_stream(step));
  const uint64_t skey = rng_key(A.sample_seed, sampler_stream(step));
  float* X = smem + S.x;
  float* H1 = smem + S.h1;
  float* H2 = smem + S.h2;
  float* D3 = smem + S.d3;
  uint8_t* meta = reinterpret_cast<uint8_t*>(smem + S.meta);
  float aw1[4][8] = {}, aw2[4][8] = {}, aw3[1][8] = {}, ab = 0.f, ab3 = 0.f;
  float loss_acc = 0.f;

  for (int64_t base = (int64_t)blockIdx.x * kBTile; base < A.n; base += (int64_t)gridDim.x * kBTile) {
    // ---- texel (one per lane, the same in every warp) -> rows ----------------
    {
      const int64_t i = base + lane;
      const bool valid = i < A.n;
      int x = 0, y = 0, m = 0;
      if (valid) {
        if (A.uvl) query_texel(M, A.uvl[3 * i], A.uvl[3 * i + 1], A.uvl[3 * i + 2], x, y, m);
        else sample_train_texel(A.crops != 0, skey, i, M.width, M.height, M.mips, x, y, m);
      }
      ColumnSink sink{X + lane};
      if (warp < 2) {
        grid_features(M, warp, x, y, m, A.noise != 0, nkey, sink);
      } else if (warp == 2) {
        tail_features(M, x, y, m, sink);
        // the target bytes (as floats) or the upstream gradient, in D3's place
        const int wm = mip_dim(M.width, m);
        const uint8_t* trow = A.train ? A.target + A.tgt_off[m] + ((int64_t)y * wm + x) * C : nullptr;
#pragma unroll 4
        for (int c = 0; c < kMaxC; ++c)
          D3[c * kLd + lane] = valid && c < C ? (A.train ? (float)trow[c] : A.dout[i * C + c]) : 0.f;
      } else {
        // cell addresses and weights of the texel's taps in both grids
        float** ga = reinterpret_cast<float**>(meta + lane * kTapMeta);
        float* wt = reinterpret_cast<float*>(meta + lane * kTapMeta + 64);
        const int j = level_of_mip(m, M.levels);
        const int wm = mip_dim(M.width, m), hm = mip_dim(M.height, m);
        const ntc_level& Lv = M.lv[j];
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          float* g = k ? A.g.grid1[j] : A.g.grid0[j];
          const Taps t = bilinear_taps(x, y, wm, hm, k ? Lv.g1_w : Lv.g0_w, k ? Lv.g1_h : Lv.g0_h);
#pragma unroll
          for (int tp = 0; tp < 4; ++tp) {
            ga[4 * k + tp] = g && valid ? g + (size_t)t.cell[tp] * (k ? M.c1 : M.c0) : nullptr;
            wt[4 * k + tp] = (k == 0 && learned0 ? 1.f : t.w[tp]) * A.grad_scale;
          }
        }
      }
    }
    __syncthreads();
    // ---- forward -------------------------------------------------------------
    float2 z[4][2], g1[4][2], g2[4][2];
    auto bias = [&](const float* b) {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float v = b ? b[ng + 16 * j] : 0.f;
        z[j][0] = z[j][1] = make_float2(v, v);
      }
    };
    bias(smem + S.b1);
    tile_dense(smem + S.w1f, X, K, ng, qg, z);
    activate(M.act, z, g1);
    put_units(H1, ng, qg, z);
    __syncthreads();
    bias(smem + S.b2);
    tile_dense(smem + S.w2f, H1, kHidden, ng, qg, z);
    activate(M.act, z, g2);
    put_units(H2, ng, qg, z);
    __syncthreads();
    {
      // output channel ng of four texels; loss and D3
      float o[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) o[e] = smem[S.b3 + ng];
#pragma unroll 4
      for (int k = 0; k < kHidden; ++k) {
        const float4 h = *reinterpret_cast<const float4*>(H2 + k * kLd + 4 * qg);
        const float w = smem[S.w3f + k * kMaxC + ng];
        o[0] = fmaf(w, h.x, o[0]);
        o[1] = fmaf(w, h.y, o[1]);
        o[2] = fmaf(w, h.z, o[2]);
        o[3] = fmaf(w, h.w, o[3]);
      }
      float4* dp = reinterpret_cast<float4*>(D3 + ng * kLd + 4 * qg);
      const float4 t4 = *dp;
      const float tv[4] = {t4.x, t4.y, t4.z, t4.w};
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        float g = 0.f;
        if (base + 4 * qg + e < A.n && ng < C) {
          const float yc = out_fwd(M.out_act, o[e]);
          float dy;
          if (A.train) {
            const float er = yc - tv[e] * (1.f / 255.f);
            loss_acc = fmaf(er, er, loss_acc);
            dy = 2.f * er;
          } else {
            dy = tv[e];
          }
          g = M.out_act == NTC_OUT_IDENTITY ? dy : dy * yc * (1.f - yc);
        }
        o[e] = g;
      }
      *dp = make_float4(o[0], o[1], o[2], o[3]);
    }
    __syncthreads();
    // ---- output layer: dW3, db3, D2 over H2 ------------------------------------
    outer_acc<1>(D3, H2, og, ig, kHidden, aw3);
    if (tid < kMaxC) ab3 += row_sum(D3 + tid * kLd);
    bias(nullptr);
    tile_dense(smem + S.w3b, D3, kMaxC, ng, qg, z);
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int p = 0; p < 2; ++p) z[j][p] = make_float2(z[j][p].x * g2[j][p].x, z[j][p].y * g2[j][p].y);
    __syncthreads();  // H2 read
    put_units(H2, ng, qg, z);
    __syncthreads();
    // ---- layer 2: dW2, db2, D1 over H1 -----------------------------------------
    outer_acc<4>(H2, H1, og, ig, kHidden, aw2);
    if (tid >= kHidden) ab += row_sum(H2 + (tid - kHidden) * kLd);
    bias(nullptr);
    tile_dense(smem + S.w2b, H2, kHidden, ng, qg, z);
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int p = 0; p < 2; ++p) z[j][p] = make_float2(z[j][p].x * g1[j][p].x, z[j][p].y * g1[j][p].y);
    __syncthreads();  // H1 and D2 read
    put_units(H1, ng, qg, z);
    __syncthreads();
    // ---- layer 1: dW1, db1, dX (over D2) ----------------------------------------
    outer_acc<4>(H1, X, og, ig, K, aw1);
    if (tid < kHidden) ab += row_sum(H1 + tid * kLd);
    if (A.grids) {
      bias(nullptr);
      tile_dense(smem + S.w1b, H1, kHidden, ng, qg, z);
      put_units(H2, ng, qg, z);
      __syncthreads();
      // each warp scatters eight texels: lane j adds grid j / 16, tap
      // (j / 4) % 4, four channels at a time, so the four lanes of a tap
      // reduce 64 consecutive bytes of one cell
      const int k = lane >> 4, slot = lane >> 2, qd = lane & 3;
      const int c = k ? M.c1 : M.c0;
      const int col = k ? W0 : (learned0 ? (slot & 3) * c : 0);
      const float* dx = H2 + col * kLd;
#pragma unroll 2
      for (int t = 8 * warp; t < 8 * warp + 8; ++t) {
        float* const ga = *reinterpret_cast<float* const*>(meta + t * kTapMeta + 8 * slot);
        if (!ga) continue;
        const float w = *reinterpret_cast<const float*>(meta + t * kTapMeta + 64 + 4 * slot);
        if ((c & 3) == 0) {
          for (int ch = 4 * qd; ch < c; ch += 16)
            atomicAdd(reinterpret_cast<float4*>(ga + ch),
                      make_float4(dx[ch * kLd + t] * w, dx[(ch + 1) * kLd + t] * w,
                                  dx[(ch + 2) * kLd + t] * w, dx[(ch + 3) * kLd + t] * w));
        } else {
          for (int ch = qd; ch < c; ch += 4) atomicAdd(ga + ch, dx[ch * kLd + t] * w);
        }
      }
    }
    __syncthreads();  // tile buffers free
  }

  // ---- flush: the CTA's weight gradients row-major over the weights' place ------
  // The grid is a whole number of clusters, so its last CTAs may have no tile:
  // they come here straight from the transposes, whose writes the staging
  // below runs over.
  __syncthreads();
  const float gs = A.grad_scale;
  float* f1 = smem;                        // [64][K]
  float* f2 = f1 + kHidden * K;            // [64][64]
  float* f3 = f2 + kHidden * kHidden;      // [16][64]
  float* fb = f3 + kMaxC * kHidden;        // db1, db2, db3
#pragma unroll
  for (int s = 0; s < 8; ++s) {
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      if (8 * s < K) f1[(og + 16 * r) * K + ig + 8 * s] = aw1[r][s];
      f2[(og + 16 * r) * kHidden + ig + 8 * s] = aw2[r][s];
    }
    f3[og * kHidden + ig + 8 * s] = aw3[0][s];
  }
  fb[tid] = ab;
  if (tid < kMaxC) fb[2 * kHidden + tid] = ab3;
  const bool loss = A.train && A.loss;
  if (loss) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) loss_acc += __shfl_xor_sync(0xffffffffu, loss_acc, o);
    if (lane == 0) smem[S.red + warp] = loss_acc;
  }
  // Two CTAs an SM come in clusters of two, which add their gradients before
  // one reduction into memory: so many CTAs each round the running totals that
  // with a reduction of each CTA's own the weight gradients of 2^15 to 2^18
  // texels were 2.2e-7 to 3e-7 from 64 bits, against 1.6e-7 to 2.2e-7.
  auto cluster = cooperative_groups::this_cluster();
  const int rank = cluster.block_rank();
  const bool pair = cluster.num_blocks() == 2;
  if (pair) cluster.sync();
  else __syncthreads();
  const float* mate = pair ? cluster.map_shared_rank(smem, rank ^ 1) : nullptr;
#pragma unroll 1
  for (int l = 0; l < 6; ++l) {  // rolled: the code is fetched cold
    float* g = l < 3 ? A.g.w[l] : A.g.b[l - 3];
    const float* src = l == 0 ? f1 : (l == 1 ? f2 : (l == 2 ? f3 : fb + (l - 3) * kHidden));
    const int n = l == 0 ? kHidden * K : (l == 1 ? kHidden * kHidden : (l == 2 ? C * kHidden : (l == 5 ? C : kHidden)));
    flush_rows(g, src, pair ? mate + (src - smem) : nullptr, rank, n, gs);
  }
  if (loss && !pair) cluster.sync();
  if (loss && tid == 0 && rank == 0) {
    // the losses too: the running total is rounded once per 128 (64) texels
    float sum = 0.f;
    for (unsigned k = 0; k < cluster.num_blocks(); ++k) {
      const float* red = cluster.map_shared_rank(smem + S.red, k);
      sum += (red[0] + red[1] + red[2] + red[3]) * A.loss_scale;
    }
    atomicAdd(A.loss, sum);
  }
  if (pair || loss) cluster.sync();  // no CTA leaves while another reads its rows
}

}  // namespace

namespace {
// Warps per CTA of the tiled forward: the most (16, 12, 8 or 4) whose
// activations fit beside the weights (16 up to K = 64, 12 at K = 96 with two
// hidden layers, 8 at K = 128).
int simt_warps(const SW& L) {
  for (int w = kMaxWarps; w > 4; w -= 4)
    if (L.bytes(w) <= 227 * 1024) return w;
  return 4;
}
// One CTA per SM; tile t goes to CTA t mod grid, so a call with fewer tiles
// than warps spreads over all SMs.
int simt_grid(int64_t n) {
  const int64_t tiles = (n + 31) / 32, cap = sm_count();
  return (int)(tiles < cap ? tiles : cap);
}
}  // namespace

cudaError_t launch_decode_simt(const ntc_material& m, const float* uvl, int64_t n, void* out,
                               int out_dtype, int filter, int noise, uint64_t noise_seed,
                               int64_t noise_step, cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  const uint64_t nkey = rng_key(noise_seed, noise_stream(noise_step));
  const uint64_t jkey = jitter_key(noise_seed, noise_step);
  const SW L(m.k_in, m.hidden_layers == 3);
  const int warps = simt_warps(L);
  const size_t smem = L.bytes(warps);
  const cudaError_t e = cudaFuncSetAttribute(
      decode_simt_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  decode_simt_kernel<<<simt_grid(n), 32 * warps, smem, s>>>(m, uvl, n, out, out_dtype, filter, noise,
                                                            nkey, jkey);
  return cudaGetLastError();
}

cudaError_t launch_f8_calibrate(const ntc_material& m, const float* uvl, int64_t n,
                               uint32_t* amax, float* sa, cudaStream_t s) {
  cudaError_t e = cudaMemsetAsync(amax, 0, 3 * sizeof(uint32_t), s);
  if (e != cudaSuccess) return e;
  if (n > 0) {
    const SW L(m.k_in, false);
    const int warps = simt_warps(L);
    const size_t smem = L.bytes(warps);
    e = cudaFuncSetAttribute(f8_calib_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    f8_calib_kernel<<<simt_grid(n), 32 * warps, smem, s>>>(m, uvl, n, amax);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  f8_scales_kernel<<<1, 32, 0, s>>>(amax, sa);
  return cudaGetLastError();
}

cudaError_t launch_backward_simt(const ntc_material& m, const BwdArgs& a, cudaStream_t s) {
  if (a.n == 0) return cudaSuccess;
  const SB S(m.k_in);
  const size_t smem = (size_t)S.size * sizeof(float);
  cudaError_t e = cudaFuncSetAttribute(backward_simt_kernel,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const int64_t tiles = (a.n + kBTile - 1) / kBTile;
  const int64_t cap = 2 * (int64_t)sm_count();
  const int64_t grid = tiles < cap ? tiles : cap;
  // With two CTAs per SM clusters of four no longer find room for the whole
  // grid at once (2^18 texels 451 -> 749 us), clusters of two do.
  const unsigned cl = grid <= sm_count() ? kBCluster : 2;
  cudaLaunchAttribute at = {};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = cl;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)((grid + cl - 1) / cl * cl));
  cfg.blockDim = dim3(kBThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, backward_simt_kernel, m, a);
}

}  // namespace ntc
