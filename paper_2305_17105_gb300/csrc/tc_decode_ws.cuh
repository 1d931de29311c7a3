// Warp-specialised tensor-core decode kernel (FP16 and FP8-E4M3), shared by
// the translation units that instantiate it: every fast-layout class of the
// FP16 form in tc_decode_ws.cu, the FP8 form in tc_decode_ws_f8.cu.
#pragma once
#include "tc_decode_common.cuh"

namespace ntc {

namespace {

// ---------------------------------------------------------------------------
// Warp-specialised form (FP16 or FP8-E4M3): five compute warpgroups, each
// running its own stream of tiles, and issuer warps, of which warp w issues
// every tcgen05.mma chain of compute warpgroup w.  A chain of dependent MMAs holds
// its issuing thread until it drains, so issuing from the compute warps
// stalls them; here they only hand over through mbarriers and keep working:
//   X(i) in shared memory --x--> L1 --d--> epilogue 1 -> H --h--> L2 --d-->
//   epilogue 2 -> H --h--> L3 (own accumulator D3) --o--> output,
// and while L2(i) runs the compute warps build X(i+1), while L3(i) runs they
// gather the cells of tile i+2, while L1(i+1) runs they write tile i.  L1
// reads its A operand from shared memory, the bias steps a constant-one A
// block in shared memory; L2 and L3 read H from TMEM.  FP8 (kind::f8f6f4):
// X and H hold E4M3 values of the layer inputs divided by their activation
// scales s_a; the epilogues apply s_w s_a and add the FP32 biases.
// TMEM per compute warpgroup (96 columns): layer 1 accumulates into [0, 64),
// and its epilogue leaves H in place in [0, 32) (a quarter of the columns is
// read before its half is written); layer 2 accumulates into [32, 96), its
// epilogue writes H over [0, 32) again; layer 3 accumulates into [80, 96),
// clear of the next tile's layer 1.  That layer's accumulator covers the H
// which layer 3 reads, and two MMAs are ordered by themselves only where they
// share accumulator and shape: the issuer waits for layer 3's commit before
// it issues the next layer 1.
//
// What bounds it: the latency of a tile's chain of stages, of which the warps
// in flight hide part (issue slots half used, L1 three quarters).  96 columns
// instead of 112 let a fifth pipeline in, and the issuers keep a chain's
// steps 43 cycles apart (tc::elect_one): 2^24 random queries of a 4096^2 x 16
// material 579 -> 518 us (1,450 GB/s of queries and outputs, 486 TFLOP/s), a
// trilinear 3840 x 2160 frame 2,167 -> 1,768 us, in FP8 at 1080p 694 -> 594.
// ---------------------------------------------------------------------------
constexpr int kWsCompute = 4;  // many-material kernel
constexpr int kWsThreads = kRows * (kWsCompute + 1);
// Five compute warpgroups need five issuer warps, hence a second issuer
// warpgroup; of the 72 registers that each of the 896 threads is launched
// with, the issuers pass some on: 80 per compute thread and 48 per issuer,
// or, in the lattice form, whose rows hold more cells, 88 and 32.
constexpr int kRegs5 = 72;
constexpr int compute_regs(int cls) { return cls == -2 ? 88 : 80; }
constexpr int issuer_regs(int cls) { return cls == -2 ? 32 : 48; }
static_assert(5 * compute_regs(5) + 2 * issuer_regs(5) <= 7 * kRegs5 &&
                  5 * compute_regs(-2) + 2 * issuer_regs(-2) <= 7 * kRegs5,
              "the warpgroups' shares fit the registers the block is launched with");
constexpr int ws_threads(int nc) { return kRows * (nc + (nc > 4 ? 2 : 1)); }
constexpr uint32_t kWsCols = 96, kWsD2 = 32, kWsD3 = 80;  // TMEM columns
constexpr int kColD3 = 96;  // many-material kernel
constexpr int kLattice = -2;
enum { kWsPlain, kWsRows, kWsTri, kWsStoch };

struct WsPlan {
  uint32_t cst, x, xbytes, stage, total;
  // stage: output rows of every compute warp (32 C floats) of the ROWS form
  __host__ __device__ WsPlan(const Plan& P, bool f8, int nc, int C, bool rows) {
    uint32_t o = (P.total + 1023) / 1024 * 1024;
    cst = o;  o += kRows * 16 * 2;                 // constant-one A block (K = 16, FP16)
    xbytes = kRows * P.k_int * (f8 ? 1 : 2);
    x = o;    o += nc * xbytes;                    // one X tile per compute warpgroup
    stage = o;
    o += rows ? nc * kRows * C * 4 : 0;
    total = o;
  }
};

// FP8 input rows: the FP16 groups the builders produce, divided by the
// layer-1 activation scale and rounded to E4M3 (saturating), 8 bytes a group.
struct F8Row {
  SmemRow dst;
  __half2 inv;
  __device__ __forceinline__ uint32_t cv(uint32_t a, uint32_t b) const {
    return tc::h2_to_e4m3x2(h2u(__hmul2(u2h(a), inv))) |
           (tc::h2_to_e4m3x2(h2u(__hmul2(u2h(b), inv))) << 16);
  }
  __device__ __forceinline__ void put4(int g, uint4 w) const { dst.put2(g, cv(w.x, w.y), cv(w.z, w.w)); }
  __device__ __forceinline__ void put2(int g, uint32_t a, uint32_t b) const { dst.put2(g, a, b); }
};

// FP8 hidden-layer epilogue in quarters, in the next layer's input units:
// z' = (s_w s_a / s_a') acc + b / s_a' (paired FMAs; `bias` holds b / s_a'),
// then act(z) / s_a' = max(z', 0) (folded into the E4M3 conversion) or, for
// hardGELU, z' sat(z' s_a' / 3 + 1/2); E4M3 into the A row (TMEM, four
// values per column).
__device__ __forceinline__ void hidden_epilogue_q8(uint32_t td, uint32_t ta, int act,
                                                   const float* bias, float scale, float hk) {
  const float2 sc2 = make_float2(scale, scale);
#pragma unroll
  for (int qtr = 0; qtr < 4; ++qtr) {
    float a[16];
    tc::tmem_ld16(td + 16 * qtr, a);
    tc::tmem_ld_wait();
    const float2* b2 = reinterpret_cast<const float2*>(bias + 16 * qtr);
    uint32_t e[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const float2 z = __ffma2_rn(make_float2(a[2 * i], a[2 * i + 1]), sc2, b2[i]);
      e[i] = act == NTC_ACT_RELU
                 ? tc::pack_e4m3x2_relu(z.x, z.y)
                 : tc::pack_e4m3x2(z.x * __saturatef(fmaf(z.x, hk, 0.5f)),
                                   z.y * __saturatef(fmaf(z.y, hk, 0.5f)));
    }
    tc::tmem_st4(ta + 4 * qtr, make_uint4(e[0] | (e[1] << 16), e[2] | (e[3] << 16),
                                          e[4] | (e[5] << 16), e[6] | (e[7] << 16)));
  }
}

// H3: a third hidden layer (FP16).  MODE: nearest texels, the outputs stored
// by the row's thread (kWsPlain) or, for channel counts that are not multiples
// of four, through shared memory (kWsRows); trilinear (kWsTri) or stochastic
// filtering (kWsStoch).  Each is a kernel of its own: with the filter read at
// run time the nearest decode's loop spilled (2^24 queries 531 -> 581 us).  NC:
// compute warpgroups, 5 for the layouts known at compile time and the lattice
// form, 4 for those read from the plan.
template <int CLS, bool F8, bool H3, int MODE, int NC>
__global__ void __launch_bounds__(ws_threads(NC), 1) decode_ws_kernel(
    const ntc_material M, const float* __restrict__ uvl, int64_t n, void* __restrict__ out,
    int out_dtype, uint64_t jkey, int* status) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  __shared__ uint64_t bar_x[NC], bar_h[NC], bar_d[NC],
      bar_o[NC], bar_r[NC], bar_fin[NC];
  __shared__ uint32_t tmem_base;
  __shared__ int wg_abort[NC];
  // CLS > 0: compile-time fast class; -1: fast layout with the class read
  // from the plan (learned interpolation); 0: generic layout; kLattice: the
  // generic layout's rows built on the integer lattice
  constexpr bool FAST = CLS > 0 || CLS == -1;
  const Plan P(M, F8, FAST);
  const WsPlan W(P, F8, NC, M.channels, MODE == kWsRows);
  uint8_t* sm = smem_raw;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int wg = warp >> 2, row = tid & (kRows - 1);

  stage_shared<F8>(M, P, sm, tid, blockDim.x);
  // constant-one A block: every row (1, 1, 0, ..., 0)
  for (int i = tid; i < kRows * 16 / 2; i += blockDim.x) {
    const int chunk = i >> 2, e = i & 3;
    reinterpret_cast<uint32_t*>(sm + W.cst)[i] =
        (chunk < kRows && e == 0) ? tc::pack_f16x2(1.f, 1.f) : 0u;
  }
  if (warp == 0) {
    tc::tmem_alloc(&tmem_base, 512);
    tc::tmem_relinquish();
  }
  if (tid < NC) {
    tc::mbar_init(&bar_x[tid], 4);
    tc::mbar_init(&bar_h[tid], 4);
    tc::mbar_init(&bar_d[tid], 1);
    tc::mbar_init(&bar_o[tid], 1);
    tc::mbar_init(&bar_r[tid], 4);
    tc::mbar_init(&bar_fin[tid], 1);
    wg_abort[tid] = 0;
  }
  if (wg < NC) zero_tail_groups<F8>(P, SmemRow{smem_row(sm + W.x + wg * W.xbytes, row)});
  tc::fence_mbar_init();
  tc::fence_proxy_async();
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  if (F8) {
    // hidden biases in the next layer's input units: b / s_a'
    float* b = reinterpret_cast<float*>(sm + P.bias);
    const float i1 = 1.f / M.scale[4], i2 = 1.f / M.scale[5];
    for (int i = tid; i < kHidden; i += blockDim.x) {
      b[i] *= i1;
      b[kHidden + i] *= i2;
    }
    __syncthreads();
  }

  constexpr bool tri = MODE == kWsTri;
  constexpr int filter =
      tri ? NTC_FILTER_TRILINEAR : (MODE == kWsStoch ? NTC_FILTER_STOCHASTIC : NTC_FILTER_NEAREST);
  constexpr int per_tile = tri ? kRows / 8 : kRows;
  // tile indices fit 32 bits: 2^31 tiles' queries would be 411 GB
  const int ntiles = (int)((n + per_tile - 1) / per_tile);
  const int stride = (int)gridDim.x * NC;
  constexpr uint32_t id64 = tc::idesc(kRows, kHidden), id16 = tc::idesc(kRows, kN3);
  // the compute warpgroup served (warp-uniform for the issuers' operands)
  const int w = __shfl_sync(0xffffffffu, wg < NC ? wg : warp - 4 * NC, 0);
  const int first = (int)blockIdx.x * NC + w;
  const uint32_t tw = tmem_base + kWsCols * w;

  if (wg >= NC) {
    if (NC > 4) tc::reg_dec<issuer_regs(CLS)>();
    // ---- issuer warp w ------------------------------------------------------
    // The pipelines wait on this warp: every descriptor is an addition away
    // from a register, and the whole warp walks the tiles so that the elected
    // lane's operands are warp-uniform (tc::elect_one).
    if (w < NC) {
      constexpr int KSTEP = Cfg<F8>::KSTEP;
      constexpr uint32_t lbo = (kHidden / 8) * 128, lbo3 = (kN3 / 8) * 128;
      const uint32_t sb = tc::smem_u32(sm);
      const uint32_t xa = tc::desc_lo(sb + W.x + w * W.xbytes, 2048), cst = tc::desc_lo(sb + W.cst, 2048);
      // the tiles after W2 follow it at fixed distances (Plan)
      constexpr uint32_t EB = Cfg<F8>::EB, dw3 = kHidden * kHidden * EB, dwb2 = dw3 + kN3 * kHidden * EB;
      constexpr uint32_t dwb3 = dwb2 + kHidden * 32, dwh = dwb3 + kN3 * 32, dwbh = dwh + kHidden * kHidden * 2;
      constexpr uint32_t to3 = ((lbo3 >> 4) << 16) - ((lbo >> 4) << 16);  // the narrow tiles' stride
      const uint32_t w1 = tc::desc_lo(sb + P.w1, lbo);
      uint32_t w2 = tc::desc_lo(sb + P.w2, lbo);
      auto dsc = [](uint32_t lo) { return tc::desc_of(lo, 128); };
      const int k1 = P.k_int / KSTEP;
      // one K-step = 32 bytes of every row = two 16-byte chunk columns
      auto layer = [&](uint32_t d, uint32_t id, uint32_t b, uint32_t step, uint32_t bb, int bias,
                       uint64_t* bar) {
        if (!tc::elect_one()) return;
#pragma unroll
        for (int s = 0; s < kHidden / KSTEP; ++s) {
          if (F8) tc::mma_f8_ta(d, tw + 8 * s, dsc(b + s * step), id, s > 0);
          else tc::mma_f16_ta(d, tw + 8 * s, dsc(b + s * step), id, s > 0);
        }
        if (bias) tc::mma_f16(d, dsc(cst), dsc(bb), id, 1);
        tc::mma_commit(bar);
      };
      auto wait_all = [](uint64_t* bar, uint32_t phase) {
        return __all_sync(0xffffffffu, tc::mbar_wait(bar, phase, kWaitLimit)) != 0;
      };
      uint32_t px = 0, ph = 0;
      bool ok = true;
      for (int tl = first; tl < ntiles; tl += stride) {
        asm volatile("" : "+r"(w2));  // form the descriptors below anew: hoisted, they would spill
        if (!(ok = wait_all(&bar_x[w], px))) break;
        // the previous tile's layer 3 no longer reads H (trilinear: and its
        // output has been read)
        if (tl != first && !(ok = wait_all(tri ? &bar_r[w] : &bar_o[w], px ^ 1))) break;
        px ^= 1;
        tc::fence_after_sync();
        if (tc::elect_one()) {
#pragma unroll 2
          for (int s = 0; s < k1; ++s) {
            if (F8) tc::mma_f8(tw, dsc(xa + 256 * s), dsc(w1 + 128 * s), id64, s > 0);
            else tc::mma_f16(tw, dsc(xa + 256 * s), dsc(w1 + 128 * s), id64, s > 0);
          }
          tc::mma_commit(&bar_d[w]);
        }
        if (!(ok = wait_all(&bar_h[w], ph))) break;
        ph ^= 1;
        tc::fence_after_sync();
        layer(tw + kWsD2, id64, w2, 128, w2 + dwb2 / 16, !F8, &bar_d[w]);
        if (H3) {
          // third hidden layer, like layer 2
          if (!(ok = wait_all(&bar_h[w], ph))) break;
          ph ^= 1;
          tc::fence_after_sync();
          layer(tw + kWsD2, id64, w2 + dwh / 16, 128, w2 + dwbh / 16, 1, &bar_d[w]);
        }
        if (!(ok = wait_all(&bar_h[w], ph))) break;
        ph ^= 1;
        tc::fence_after_sync();
        layer(tw + kWsD3, id16, w2 + dw3 / 16 + to3, 32, w2 + dwb3 / 16 + to3, !F8, &bar_o[w]);
      }
      if (!ok) *reinterpret_cast<volatile int*>(&wg_abort[w]) = 1;
      // every MMA of this thread completes before TMEM is released
      if (tc::elect_one()) tc::mma_commit(&bar_fin[w]);
      if (!tc::mbar_wait(&bar_fin[w], 0, kWaitLimit)) *reinterpret_cast<volatile int*>(&wg_abort[w]) = 1;
    }
  } else {
    if (NC > 4) tc::reg_inc<compute_regs(CLS)>();
    // ---- compute warpgroup w -------------------------------------------------
    const uint32_t lq = (uint32_t)((warp & 3) * 32) << 16;
    const uint32_t td = tw + lq, td2 = tw + kWsD2 + lq, td3 = tw + kWsD3 + lq;
    const SmemRow xs{smem_row(sm + W.x + w * W.xbytes, row)};
    const MipTab* tb = reinterpret_cast<const MipTab*>(sm + P.tab);
    const FastK K(M);
    const LatticeK KL(M);
    auto gather = [&](Row& r) {
      if (CLS > 0) gather_fast(FastLayout<(CLS > 0 ? CLS : 1)>(), tb, r);
      else if (CLS == kLattice) gather_lattice(P, tb, r);
      else if (CLS < 0) gather_fast(P, tb, r);
    };
    volatile int* abort_flag = &wg_abort[w];
    // FP8: per-layer accumulator scales s_w s_a (layer 3 pre-halved for the
    // tanh form of the sigmoid) and inverse activation scales
    float sc[3] = {1.f, 1.f, 1.f}, inv_sa[3] = {1.f, 1.f, 1.f};
    if (F8) {
#pragma unroll
      for (int l = 0; l < 3; ++l) {
        sc[l] = M.scale[l] * M.scale[3 + l];
        inv_sa[l] = 1.f / M.scale[3 + l];
      }
      if (M.out_act != NTC_OUT_IDENTITY) sc[2] *= 0.5f;
    }
    const float* bias = reinterpret_cast<const float*>(sm + P.bias);
    const F8Row x8{xs, __float2half2_rn(inv_sa[0])};
    auto qindex = [&](int t) { return (int64_t)t * per_tile + (tri ? row >> 3 : row); };
    auto build = [&](const Row& r) {
      if (F8) {
        if (CLS > 0) build_fast(FastLayout<(CLS > 0 ? CLS : 1)>(), P, K, sm, r, x8);
        else build_generic<true>(M, P, sm, r, xs, inv_sa[0]);
      } else {
        if (CLS > 0) build_fast(FastLayout<(CLS > 0 ? CLS : 1)>(), P, K, sm, r, xs);
        else if (CLS == kLattice) build_lattice(M, P, KL, sm, r, xs);
        else if (CLS < 0) build_fast(P, P, K, sm, r, xs);
        else build_generic<false>(M, P, sm, r, xs, 1.f);
      }
      tc::fence_proxy_async();
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&bar_x[w]);
    };
    const int C = M.channels;
    uint32_t pd = 0, po = 0;
    int tl = first;
    int cur_valid = 0;
    float cur_wtap = 0.f;
    Row nxt;
    Query nq;
    if (tl < ntiles) {
      Row r;
      const int64_t q0 = qindex(tl);
      locate(M, tb, load_query(uvl, q0, q0 < n), filter, row, r, q0, jkey);
      gather(r);
      build(r);
      cur_valid = r.valid;
      cur_wtap = r.wtap;
      const int64_t q1 = qindex(tl + stride);
      locate(M, tb, load_query(uvl, q1, tl + stride < ntiles && q1 < n), filter, row, nxt, q1, jkey);
      gather(nxt);
      const int64_t q2 = qindex(tl + 2 * stride);
      nq = load_query(uvl, q2, tl + 2 * stride < ntiles && q2 < n);
    }
    for (; tl < ntiles; tl += stride) {
      const int64_t q = qindex(tl);
      const bool valid = cur_valid != 0;
      const float wtap = cur_wtap;
      // layer 1 -> H1
      if (!tc::mbar_wait(&bar_d[w], pd, kWaitLimit)) *abort_flag = 1;
      pd ^= 1;
      tc::fence_after_sync();
      if (F8) hidden_epilogue_q8(td, td, M.act, bias, sc[0] * inv_sa[1], M.scale[4] * (1.f / 3.f));
      else hidden_epilogue_q(td, td, M.act);
      tc::tmem_st_wait();
      tc::fence_before_sync();
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&bar_h[w]);
      // the next tile's input rows (layer 1 is done with X)
      if (tl + stride < ntiles) {
        build(nxt);
        cur_valid = nxt.valid;
        cur_wtap = nxt.wtap;
      }
      // layer 2 -> H2
      if (!tc::mbar_wait(&bar_d[w], pd, kWaitLimit)) *abort_flag = 1;
      pd ^= 1;
      tc::fence_after_sync();
      if (F8) hidden_epilogue_q8(td2, td, M.act, bias + kHidden, sc[1] * inv_sa[2], M.scale[5] * (1.f / 3.f));
      else hidden_epilogue_q(td2, td, M.act);
      tc::tmem_st_wait();
      tc::fence_before_sync();
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&bar_h[w]);
      if (H3) {
        // third hidden layer -> H
        if (!tc::mbar_wait(&bar_d[w], pd, kWaitLimit)) *abort_flag = 1;
        pd ^= 1;
        tc::fence_after_sync();
        hidden_epilogue_q(td2, td, M.act);
        tc::tmem_st_wait();
        tc::fence_before_sync();
        __syncwarp();
        if (lane == 0) tc::mbar_arrive(&bar_h[w]);
      }
      if (*abort_flag) break;
      // the tile after next: texel and cells; its successor's query
      locate(M, tb, nq, filter, row, nxt, qindex(tl + 2 * stride), jkey);
      gather(nxt);
      {
        const int t3 = tl + 3 * stride;
        const int64_t q3 = qindex(t3);
        nq = load_query(uvl, q3, t3 < ntiles && q3 < n);
      }
      // layer 3 -> output
      if (!tc::mbar_wait(&bar_o[w], po, kWaitLimit)) *abort_flag = 1;
      po ^= 1;
      tc::fence_after_sync();
      float yv[16];
      tc::tmem_ld16(td3, yv);
      tc::tmem_ld_wait();
      tc::fence_before_sync();
      if (tri) {
        // lets the next tile's layer 1 go: issued as soon as its X stands, it
        // holds up the other pipelines' layers although the blend and the
        // store still cover it (a 3840 x 2160 frame 1,994 us against 1,927;
        // with one decode a query waiting loses: 2^24 queries 547 against 557)
        __syncwarp();
        if (lane == 0) tc::mbar_arrive(&bar_r[w]);
      }
      if (F8) {
        const float2* b3 = reinterpret_cast<const float2*>(bias + 2 * kHidden);
#pragma unroll
        for (int c = 0; c < 16; c += 2) {
          const float2 z = __ffma2_rn(make_float2(yv[c], yv[c + 1]), make_float2(sc[2], sc[2]), b3[c / 2]);
          yv[c] = z.x;
          yv[c + 1] = z.y;
        }
      }
      out_activate(yv, M.out_act);
      if (tri) {
        const int c = blend_taps(yv, wtap, row);
        if (valid) store_pair(out, out_dtype, q * C, C, c, yv[0], yv[1]);
      } else if (MODE == kWsRows) {
        const int rows = __popc(__ballot_sync(0xffffffffu, valid));
        float* st = reinterpret_cast<float*>(sm + W.stage) + (warp * 32) * C;
        store_rows(st, out, out_dtype, (q - lane) * C, rows, C, lane, yv);
      } else if (valid) {
        store_texel(out, out_dtype, q, C, yv);
      }
      if (*abort_flag) break;
    }
  }

  tc::fence_before_sync();
  __syncthreads();
  if (tid == 0) {
    int any = 0;
    for (int i = 0; i < NC; ++i) any |= wg_abort[i];
    if (any) atomicExch(status, NTC_ERR_TIMEOUT);
  }
  if (warp == 0) {
    tc::fence_after_sync();
    tc::tmem_dealloc(tmem_base, 512);
  }
}

template <int CLS, bool F8, bool H3, int MODE, int NC>
cudaError_t launch_ws_nc(const ntc_material& m, const float* uvl, int64_t n, void* out,
                         int out_dtype, int filter, uint64_t jkey, cudaStream_t s) {
  const Plan P(m, F8, CLS > 0 || CLS == -1);
  if (P.h3 != H3) return cudaErrorInvalidValue;
  const WsPlan W(P, F8, NC, m.channels, MODE == kWsRows);
  auto* kernel = decode_ws_kernel<CLS, F8, H3, MODE, NC>;
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)W.total);
  if (e != cudaSuccess) return e;
  const int per_tile = filter == NTC_FILTER_TRILINEAR ? kRows / 8 : kRows;
  const int64_t tiles = (n + per_tile - 1) / per_tile;
  const int64_t ctas = (tiles + NC - 1) / NC;
  const int64_t cap = sm_count();
  const int grid = (int)(ctas < cap ? ctas : cap);
  kernel<<<grid, ws_threads(NC), W.total, s>>>(m, uvl, n, out, out_dtype, jkey, status_word());
  return cudaGetLastError();
}

template <int CLS, bool F8, int MODE, bool H3 = false>
cudaError_t launch_ws(const ntc_material& m, const float* uvl, int64_t n, void* out, int out_dtype,
                      int filter, uint64_t jkey, cudaStream_t s) {
  static_assert(!(F8 && H3), "three hidden layers run in FP16");
  constexpr int NC = CLS > 0 || CLS == kLattice ? 5 : 4;
  return launch_ws_nc<CLS, F8, H3, MODE, NC>(m, uvl, n, out, out_dtype, filter, jkey, s);
}

// Compile-time class of a fast-layout grid: 0 (cell of 4 bytes), 1 (9-12
// channels in 8 bytes), 2 (13-16 channels).
inline int grid_class(int c, int cb) { return cb == 4 ? 0 : (c > 12 ? 2 : 1); }

// Materials off the fast layout that take the lattice form: packed grids of 2
// or 4 bits with the fast layout's exactness conditions (other widths, F32
// grids and vector-quantised G0 blend in float), and a plan of which five
// pipelines fit beside the kernel's own 1 KB.  It does not with learned G0,
// three hidden layers and more than 16 channels in both grids (K = 144:
// 232,448 bytes); the float form's four pipelines (195,584) do.
inline bool lattice_ok(const ntc_material& m) {
  return m.encoding == NTC_GRID_PACKED && m.vq_books == 0 && (m.bits0 == 2 || m.bits0 == 4) &&
         (m.bits1 == 2 || m.bits1 == 4) && fast_layout_ok(m) &&
         WsPlan(Plan(m, false, false), false, 5, m.channels, false).total <= 226u * 1024u;
}

// The FP16 form of one mode, by layout.
template <int MODE>
cudaError_t dispatch_f16(const ntc_material& m, const float* uvl, int64_t n, void* out,
                         int out_dtype, int filter, uint64_t jkey, cudaStream_t s, bool fast) {
  const bool h3 = m.hidden_layers == 3;
#define NTC_WS(cls, third) return launch_ws<cls, false, MODE, third>(m, uvl, n, out, out_dtype, filter, jkey, s)
  if (!fast) {
    if (lattice_ok(m)) {
      if (h3) NTC_WS(kLattice, true);
      NTC_WS(kLattice, false);
    }
    if (h3) NTC_WS(0, true);
    NTC_WS(0, false);
  }
  const Plan P(m, false, true);
  const int cls = 3 * grid_class(m.c0, P.cb0) + grid_class(m.c1, P.cb1);
  if (h3) {  // a third hidden layer: the paper's profiles, else run time
    if (P.learned && cls == 5) NTC_WS(16, true);
    if (P.learned && cls == 7) NTC_WS(18, true);
    NTC_WS(-1, true);
  }
  if (P.vq) NTC_WS(-1, false);
  if (P.learned) {
    // the paper's profiles 0.5 and 2.25 (4-bit G0 of 12 / 16 channels, G1 of
    // 16 / 12) as compile-time classes, other learned layouts at run time
    if (cls == 5) NTC_WS(16, false);
    if (cls == 7) NTC_WS(18, false);
    NTC_WS(-1, false);
  }
  switch (cls) {
    case 0: NTC_WS(1, false);
    case 1: NTC_WS(2, false);
    case 2: NTC_WS(3, false);
    case 3: NTC_WS(4, false);
    case 4: NTC_WS(5, false);
    case 5: NTC_WS(6, false);
    case 6: NTC_WS(7, false);
    case 7: NTC_WS(8, false);
    default: NTC_WS(9, false);
  }
#undef NTC_WS
}

// The FP8-E4M3 form of one mode, by layout.
template <int MODE>
cudaError_t dispatch_f8(const ntc_material& m, const float* uvl, int64_t n, void* out,
                        int out_dtype, int filter, uint64_t jkey, cudaStream_t s) {
#define NTC_WS(cls) return launch_ws<cls, true, MODE>(m, uvl, n, out, out_dtype, filter, jkey, s)
  const Plan P(m, true, fast_layout_ok(m));
  if (!P.fast) NTC_WS(0);
  switch (3 * grid_class(m.c0, P.cb0) + grid_class(m.c1, P.cb1)) {
    case 0: NTC_WS(1);
    case 1: NTC_WS(2);
    case 2: NTC_WS(3);
    case 3: NTC_WS(4);
    case 4: NTC_WS(5);
    case 5: NTC_WS(6);
    case 6: NTC_WS(7);
    case 7: NTC_WS(8);
    default: NTC_WS(9);
  }
#undef NTC_WS
}

// The mode of a call.  Rows of channel counts that are not multiples of four
// pass through shared memory once a row needs many stores of its own: from 9
// FP16 or FP32 channels on (2^21 queries, FP16, C = 9: 91 -> 83 us, C = 15:
// 191 -> 86; C = 6: 83 -> 80), from 13 8-bit ones (C = 15: 99 -> 89, C = 9:
// 82 -> 85).  Where the plan with the rows takes more than 176 KB (long input
// rows: the lattice form's learned layouts) they cost the gathers their L1:
// from 11 on (C = 9: 159 -> 175, C = 15: 247 -> 179), 8-bit outputs never.
inline int ws_mode(const ntc_material& m, bool f8, bool fast, int filter, int out_dtype) {
  if (filter == NTC_FILTER_TRILINEAR) return kWsTri;
  if (filter == NTC_FILTER_STOCHASTIC) return kWsStoch;
  if ((m.channels & 3) == 0) return kWsPlain;
  const WsPlan W(Plan(m, f8, fast), f8, 5, m.channels, true);
  const bool u8 = out_dtype == NTC_DTYPE_U8, large = W.total > 176u * 1024u;
  const int least = large ? (u8 ? kMaxC + 1 : 11) : (u8 ? 13 : 9);
  return m.channels >= least && W.total <= 226u * 1024u ? kWsRows : kWsPlain;
}

}  // namespace

// One mode of the FP16 / FP8 form (a translation unit each).
cudaError_t launch_decode_ws_stoch(const ntc_material& m, const float* uvl, int64_t n, void* out,
                                   int out_dtype, int filter, uint64_t jkey, cudaStream_t s, bool fast);
cudaError_t launch_decode_ws_f8_stoch(const ntc_material& m, const float* uvl, int64_t n, void* out,
                                      int out_dtype, int filter, uint64_t jkey, cudaStream_t s);
cudaError_t launch_decode_ws_tri(const ntc_material& m, const float* uvl, int64_t n, void* out,
                                 int out_dtype, int filter, uint64_t jkey, cudaStream_t s, bool fast);
cudaError_t launch_decode_ws_rows(const ntc_material& m, const float* uvl, int64_t n, void* out,
                                  int out_dtype, int filter, uint64_t jkey, cudaStream_t s, bool fast);
cudaError_t launch_decode_ws_f8_tri(const ntc_material& m, const float* uvl, int64_t n, void* out,
                                    int out_dtype, int filter, uint64_t jkey, cudaStream_t s);
cudaError_t launch_decode_ws_f8_rows(const ntc_material& m, const float* uvl, int64_t n, void* out,
                                     int out_dtype, int filter, uint64_t jkey, cudaStream_t s);

}  // namespace ntc
