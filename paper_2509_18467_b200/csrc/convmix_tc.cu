// Tensor-core kernels for conv -> shared linear layer -> softmax feature map (Section 4.1) and for the chain rule back
// through them (distillation step, Section 5.1), bf16 storage.
//
// Forward: one thread block = one (batch, query head, tile of 128 tokens), both streams (they share W_h), each stream's products
// behind the other one's work: depthwise causal conv in fp32 -> operand, Y = u W_h by tcgen05 (fp32 accumulator in tensor memory), phi (softmax over
// the row, or the elementwise 1 + ELU / identity of Section 2) by the threads that own the row's TMEM lane, 16-bit or fp32
// store.
// Backward (head width 64): one block = one (batch, key head, tile); for each query head of
// the group and each stream it recomputes u and p = softmax(u W_h), applies the softmax Jacobian dy = p (dp - p . dp),
// and forms du = dy W_h^T (the key stream summed over the group in registers) and dW_h += u^T dy (accumulators of two
// heads at a time in tensor memory, flushed with atomic adds). The conv's own backward then runs on du.
// Tiles are unswizzled 8x8 core matrices with every 8-column slab contiguous (see gla_tc.cu): W_h serves as the
// MN-major B of the forward mix and, without a second copy, as the K-major B of dy W_h^T.
#include <cuda.h>
#include <cuda_fp16.h>

#include <mutex>

#include "common.cuh"
#include "octet_tile.cuh"
#include "tc_common.cuh"

namespace lawcat {
namespace ctc {

struct CArgs {
  const bf16 *q, *k, *w_q, *w_k, *W, *cache_q, *cache_k;
  void *qdot, *kdot;                 // forward outputs (bf16 or fp32)
  const void *d_qdot, *d_kdot;       // backward inputs
  float *du_q, *du_k, *dW;           // backward outputs: d(conv out) per stream (fp32), dW (fp32, atomic adds)
  int* dev_status;
  int B, T, H, Hkv, K, phi;
  int unshared;  // 1: W is [2,H,D,D], the key stream mixes with the second set (forward kernel only)
};

// raw rows [t0 - HALO, t0 + TT) of one head into shared memory (rows before the sequence come from the conv cache or are
// zero, rows past its end are zero), and the head's taps as fp32 [D][4] (zero beyond the conv width)
template <int D>
__device__ __forceinline__ void load_raw_and_taps(uint8_t* s_raw, float* s_w, const bf16* x, const bf16* w, const bf16* cache,
                                                  int b, int t0, int T, int NH, int head, int K, int tid, int nthreads) {
  using L = Lay<D>;
  for (int idx = tid; idx < (TT + HALO) * L::OPR; idx += nthreads) {
    const int rr = idx / L::OPR, o = idx % L::OPR, t = t0 - HALO + rr;
    uint4 v = make_uint4(0u, 0u, 0u, 0u);
    if (t >= 0 && t < T) {
      v = *reinterpret_cast<const uint4*>(x + (((size_t)b * T + t) * NH + head) * D + o * 8);
    } else if (t < 0 && cache != nullptr && t + (K - 1) >= 0) {
      v = *reinterpret_cast<const uint4*>(cache + (((size_t)b * (K - 1) + t + (K - 1)) * NH + head) * D + o * 8);
    }
    *reinterpret_cast<uint4*>(s_raw + rr * L::RAW_STRIDE + o * 16) = v;
  }
  for (int idx = tid; idx < D * 4; idx += nthreads) {
    const int c = idx >> 2, dl = idx & 3;
    s_w[idx] = dl < K ? __bfloat162float(w[((size_t)head * D + c) * K + dl]) : 0.f;
  }
}

// depthwise causal conv of the tile in fp32, result as the fp16 A operand of the mix; s_ul (nullable): the low part
// u - fp16(u), again in fp16, for products that take u as a two-term operand
template <int D>
__device__ __forceinline__ void conv_tile(const uint8_t* s_raw, const float* s_w, uint8_t* s_u, int tid, int nthreads,
                                          uint8_t* s_ul = nullptr) {
  using L = Lay<D>;
  const int o = tid % L::OPR;
  float w[8][4];
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const float4 t4 = *reinterpret_cast<const float4*>(s_w + (o * 8 + i) * 4);
    w[i][0] = t4.x; w[i][1] = t4.y; w[i][2] = t4.z; w[i][3] = t4.w;
  }
#pragma unroll 1
  for (int r = tid / L::OPR; r < TT; r += nthreads / L::OPR) {
    float u[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int dl = 0; dl < 4; ++dl) {
      float x[8];
      unpack8b(*reinterpret_cast<const uint4*>(s_raw + (r + HALO - dl) * L::RAW_STRIDE + o * 16), x);
#pragma unroll
      for (int i = 0; i < 8; ++i) u[i] = fmaf(w[i][dl], x[i], u[i]);
    }
    const uint4 ph = pack8f16(u);
    *reinterpret_cast<uint4*>(s_u + toff(L::SLAB_U, r, o * 8)) = ph;
    if (s_ul != nullptr) {
      const __half2* h2 = reinterpret_cast<const __half2*>(&ph);
      float lo[8];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float2 f = __half22float2(h2[i]);
        lo[2 * i] = u[2 * i] - f.x;
        lo[2 * i + 1] = u[2 * i + 1] - f.y;
      }
      *reinterpret_cast<uint4*>(s_ul + toff(L::SLAB_U, r, o * 8)) = pack8f16(lo);
    }
  }
}

// Forward. One block (16 warps per SM) walks one (batch, query head, tile of 128 tokens), query stream then key stream. bf16 outputs take
// the conv output as one fp16 operand. fp32 outputs (features that a fused caller keeps in fp32, and those of the exact
// recurrence) take it as three bf16 terms, u = b1 + b2 + b3 exactly, with W_h exact in bf16: the products are those of
// fp32 numbers over the full fp32 range, summed in fp32.
// Bound by instruction issue and the dependent phases of a tile. The products run behind other work: the key stream's conv (into
// registers) while the query stream's mix runs, the query stream's features and their way out while the key stream's does. Outputs
// leave through a staging tile as whole rows. fp32 outputs, 32/8 heads, against one stream after the other: 4 x 1300 tokens of 128
// channels 148 -> 134 us, 8 x 1024 of 64 84 -> 76, 4096 of 128 107 -> 99.
template <int D, typename TO>
__host__ __device__ constexpr int fwd_threads() { return D == 128 && sizeof(TO) == 4 ? 512 : 256; }
template <int D, typename TO>
struct FwdMap {  // shared memory
  using L = Lay<D>;
  static constexpr int NT = sizeof(TO) == 4 ? 3 : 1, NCG = fwd_threads<D, TO>() / 128;
  static constexpr uint32_t WT = 0, U = WT + L::TILE_W, ST = U + NT * L::TILE_U, TAPS = ST + TT * D * sizeof(TO);
  static constexpr uint32_t RED = TAPS + 2 * D * 16, BAR = RED + NCG * TT * 4, BYTES = BAR + 64;
};

template <int D, typename TO>
__global__ void __launch_bounds__(fwd_threads<D, TO>()) convmix_tc_fwd_kernel(const CArgs a) {
  using L = Lay<D>;
  using M = FwdMap<D, TO>;
  extern __shared__ __align__(128) uint8_t sg[];
  constexpr int NTH = fwd_threads<D, TO>(), NCG = M::NCG, NT = M::NT, FMT = NT == 3 ? FMT_BF16 : FMT_F16;
  const uint32_t sb = smem_u32(sg);
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;  // (warp: uniform to the compiler)
  volatile int* const s_flags = reinterpret_cast<volatile int*>(sg + M::BAR + 16);  // [0] tmem base, [1] abort
  float* const s_red = reinterpret_cast<float*>(sg + M::RED);  // [column group][128 rows]
  const int t0 = tile_of_block() * TT, bh = blockIdx.x, h = bh % a.H, b = bh / a.H;
  if (t0 >= a.T) return;
  const int G = a.H / a.Hkv, j = h / G;
  if (tid == 0) {
    mbar_init(sb + M::BAR, 1);
    mbar_fence_init();
    s_flags[1] = 0;
  }
  if (warp == 0) {
    tmem_alloc(sb + M::BAR + 16, 2 * D);
    tmem_relinquish();
  }
  asm volatile("griddepcontrol.wait;" ::: "memory");
  auto load_w = [&](const bf16* Wh) {
    if (NT == 1) {
      load_w_tile<D>(sg + M::WT, Wh, tid, NTH);
    } else {
      for (int idx = tid; idx < D * L::OPR; idx += NTH) {
        const int c = idx / L::OPR, o = idx % L::OPR;
        *reinterpret_cast<uint4*>(sg + M::WT + toff(L::SLAB_W, c, o * 8)) = *reinterpret_cast<const uint4*>(Wh + (size_t)c * D + o * 8);
      }
    }
  };
  constexpr int RPT = TT * L::OPR / NTH;  // rows of the conv per thread
  const int co = tid % L::OPR, cr0 = tid / L::OPR * RPT;
  uint4 raw[RPT + HALO];
  conv_load<D, RPT>(raw, a.q, a.cache_q, b, t0 + cr0, a.T, a.H, h, a.K, co);
  load_w(a.W + (size_t)h * D * D);
  load_taps<D>(sg + M::TAPS, a.w_q, h, a.K, tid, NTH);
  load_taps<D>(sg + M::TAPS + D * 16, a.w_k, j, a.K, tid, NTH);
  const int row = (warp & 3) * 32 + lane, cg = warp >> 2;  // epilogue: row of the tile, group of its columns
  constexpr int HC = D / NCG;
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem = (uint32_t)s_flags[0], lane_base = tmem + ((uint32_t)((warp & 3) * 32) << 16) + cg * HC;
  Waiter wt{sb + M::BAR, 0u, s_flags + 1, a.dev_status};
  auto put_u = [&](int i, uint64_t* u) {  // operand row of token cr0 + i
    uint8_t* dst = sg + M::U + toff(L::SLAB_U, cr0 + i, co * 8);
    float f[8];
    if (NT == 1) {
      pairs_to_floats(u, f);
      *reinterpret_cast<uint4*>(dst) = pack8f16(f);
    } else {
      *reinterpret_cast<uint4*>(dst) = take_bf16(u);
      *reinterpret_cast<uint4*>(dst + L::TILE_U) = take_bf16(u);
      pairs_to_floats(u, f);
      *reinterpret_cast<uint4*>(dst + 2 * L::TILE_U) = pack8bf16(f);
    }
  };
  auto mix = [&](int stream) {  // behind the operand's writes: Y = u W_h
    fence_proxy_async();
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    if (warp == 0 && elect_one()) {
      constexpr uint32_t idesc = instr_desc(128, D, FMT, MAJOR_K, MAJOR_MN);
      const uint64_t db = mview(sb + M::WT, L::SLAB_W);
#pragma unroll
      for (int term = NT - 1; term >= 0; --term) {  // (smallest terms first)
        const uint64_t da = kview(sb + M::U + term * L::TILE_U, L::SLAB_U);
#pragma unroll
        for (int kk = 0; kk < D / 16; ++kk)
          mma_f16(tmem + stream * D, dadv(da, 2 * L::SLAB_U * kk), dadv(db, 256 * kk), idesc, term < NT - 1 || kk > 0);
      }
      mma_commit(sb + M::BAR);
    }
  };
  // phi over the row: softmax (the threads of a row exchange the sum), or elementwise 1 + ELU / identity; then out
  auto features = [&](int stream) {
    float y[HC];
    auto load_y = [&]() {
#pragma unroll
      for (int c0 = 0; c0 < HC; c0 += 32) tmem_ld32(lane_base + stream * D + c0, y + c0);
      tmem_wait_ld();
    };
    load_y();
    if (a.phi == LAWCAT_PHI_SOFTMAX) {
      // While every |y| stays below Y_MAX, exp(y) needs no shift by the row's maximum, and the barrier behind which the parts of
      // the sum meet also tells whether one is missing.
      float sum, am = 0.f;
      auto exps = [&](float m) {
        sum = 0.f;
        if (NT == 3) {
#pragma unroll
          for (int i = 0; i < HC; ++i) { y[i] = expf(y[i] - m); sum += y[i]; }
        } else {
          const float mb = m * 1.4426950408889634f;
#pragma unroll
          for (int i = 0; i < HC; ++i) { y[i] = ex2f(fmaf(y[i], 1.4426950408889634f, -mb)); sum += y[i]; }
        }
      };
#pragma unroll
      for (int i = 0; i < HC; ++i) am = fmaxf(am, fabsf(y[i]));
      exps(0.f);
      s_red[cg * TT + row] = sum;
      if (__syncthreads_or(!(am < Y_MAX))) {
        __syncthreads();  // (the sums have been seen by nobody; the row's maximum takes their place)
        load_y();
        float m = -INFINITY;
#pragma unroll
        for (int i = 0; i < HC; ++i) m = fmaxf(m, y[i]);
        s_red[cg * TT + row] = m;
        __syncthreads();
#pragma unroll
        for (int i = 0; i < NCG; ++i) m = fmaxf(m, s_red[i * TT + row]);
        exps(m);
        __syncthreads();
        s_red[cg * TT + row] = sum;
        __syncthreads();
      }
      float tot = 0.f;
#pragma unroll
      for (int i = 0; i < NCG; ++i) tot += s_red[i * TT + row];
      const float inv = 1.f / tot;
#pragma unroll
      for (int i = 0; i < HC; ++i) y[i] *= inv;
    } else {
      if (a.phi == LAWCAT_PHI_ELU1) {
#pragma unroll
        for (int i = 0; i < HC; ++i) y[i] = y[i] > 0.f ? y[i] + 1.f : (NT == 3 ? expf(y[i]) : __expf(y[i]));
      }
      __syncthreads();  // (the staging tile has been read)
    }
    // rows of 16-byte pieces, XOR-swizzled, then whole rows to global memory
    constexpr int EPP = 16 / sizeof(TO), PPR = D / EPP;  // elements per piece, pieces per row
#pragma unroll
    for (int i = 0; i < HC; i += EPP) {
      const int pc = (cg * HC + i) / EPP;
      uint4 v;
      if (NT == 3) v = make_uint4(__float_as_uint(y[i]), __float_as_uint(y[i + 1]), __float_as_uint(y[i + 2]), __float_as_uint(y[i + 3]));
      else v = pack8bf16(y + i);
      *reinterpret_cast<uint4*>(sg + M::ST + (row * PPR + (pc ^ (row & 7))) * 16) = v;
    }
    __syncthreads();
    TO* out = reinterpret_cast<TO*>(stream ? a.kdot : a.qdot);
#pragma unroll 4
    for (int idx = tid; idx < TT * PPR; idx += NTH) {
      const int r = idx / PPR, pc = idx % PPR;
      if (t0 + r < a.T)
        *reinterpret_cast<uint4*>(out + (((size_t)b * a.T + t0 + r) * a.H + h) * D + pc * EPP) =
            *reinterpret_cast<const uint4*>(sg + M::ST + (r * PPR + (pc ^ (r & 7))) * 16);
    }
  };
  conv_emit<D, RPT>(raw, sg + M::TAPS, co, put_u);
  mix(0);
  uint64_t uk[RPT][4];
  conv_load<D, RPT>(raw, a.k, a.cache_k, b, t0 + cr0, a.T, a.Hkv, j, a.K, co);
  conv_emit<D, RPT>(raw, sg + M::TAPS + D * 16, co, [&](int i, uint64_t* u) {
#pragma unroll
    for (int c = 0; c < 4; ++c) uk[i][c] = u[c];
  });
  wt.wait();  // (the operand tile, and W_h, have been read)
#pragma unroll
  for (int i = 0; i < RPT; ++i) put_u(i, uk[i]);
  if (a.unshared) load_w(a.W + ((size_t)a.H + h) * D * D);  // (a separate linear layer per stream)
  mix(1);
  features(0);
  wt.wait();
  features(1);
  tc_fence_before_sync();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after_sync();
    tmem_dealloc(tmem, 2 * D);
  }
}

// Backward through phi and the mix for head width 64: du_q [B,T,H,64], du_k [B,T,Hkv,64] (fp32), dW [H,64,64] (atomic adds
// into a zeroed array).
__global__ void __launch_bounds__(128, 2) convmix_tc_bwd_kernel(const CArgs a) {
  typedef bf16 TG;  // of the incoming gradients
  constexpr int D = 64;
  using L = Lay<D>;
  extern __shared__ __align__(128) uint8_t sg[];
  constexpr uint32_t OFF_WT = 0, OFF_U = OFF_WT + L::TILE_W, OFF_DY = OFF_U + L::TILE_U, OFF_DYL = OFF_DY + L::TILE_U;
  constexpr uint32_t OFF_UL = OFF_DYL + L::TILE_U;  // low part of the conv output (second term of u in dW)
  constexpr uint32_t OFF_RAW = OFF_UL + L::TILE_U + 2048, OFF_TAPS = OFF_RAW + (L::RAW_BYTES + 15) / 16 * 16;
  constexpr uint32_t OFF_BAR = OFF_TAPS + D * 4 * 4;
  constexpr uint32_t COL_Y = 0, COL_DW = 64, TMEM_COLS = 256;  // Y / du, and the dW accumulators of two heads at a time
  const uint32_t sb = smem_u32(sg);
  const int tid = threadIdx.x, warp = tid >> 5;
  volatile int* const s_flags = reinterpret_cast<volatile int*>(sg + OFF_BAR + 16);
  const int t0 = tile_of_block() * TT, bj = blockIdx.x, j = bj % a.Hkv, b = bj / a.Hkv;
  if (t0 >= a.T) return;
  const int G = a.H / a.Hkv;
  if (tid == 0) {
    mbar_init(sb + OFF_BAR, 1);
    mbar_fence_init();
    s_flags[1] = 0;
  }
  if (warp == 0) {
    tmem_alloc(sb + OFF_BAR + 16, TMEM_COLS);
    tmem_relinquish();
  }
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem = (uint32_t)s_flags[0];
  const uint32_t lane_base = tmem + ((uint32_t)(warp * 32) << 16);
  Waiter wt{sb + OFF_BAR, 0u, s_flags + 1, a.dev_status};
  const int t = t0 + tid;       // the row this thread owns in the epilogues
  const bool valid = t < a.T;
  float duk[D];                 // d(conv out) of the key stream, summed over the heads of the group
#pragma unroll
  for (int i = 0; i < D; ++i) duk[i] = 0.f;
#pragma unroll 1
  for (int g = 0; g < G; ++g) {
    const int h = j * G + g;
    load_w_tile<D>(sg + OFF_WT, a.W + (size_t)h * D * D, tid, 128);
#pragma unroll 1
    for (int stream = 0; stream < 2; ++stream) {
      const bf16* x = stream ? a.k : a.q;
      const int NH = stream ? a.Hkv : a.H, head = stream ? j : h;
      load_raw_and_taps<D>(sg + OFF_RAW, reinterpret_cast<float*>(sg + OFF_TAPS), x, stream ? a.w_k : a.w_q,
                           stream ? a.cache_k : a.cache_q, b, t0, a.T, NH, head, a.K, tid, 128);
      if (valid) {
        // towards L2 while conv and mix run: this thread's row of the incoming gradient (read in the epilogue below),
        // and its raw row of the next (head, stream) step
        const char* dpr = reinterpret_cast<const char*>(stream ? a.d_kdot : a.d_qdot) +
                          ((((size_t)b * a.T + t) * a.H + h) * D) * sizeof(TG);
        prefetch_l2(dpr);
        if (sizeof(TG) * D > 128) prefetch_l2(dpr + 128);
        const int ns = stream ^ 1, ng = g + stream;  // the step that follows
        if (ng < G) {
          const bf16* nx = ns ? a.k : a.q;
          const int nNH = ns ? a.Hkv : a.H, nhead = ns ? j : j * G + ng;
          prefetch_l2(nx + (((size_t)b * a.T + t) * nNH + nhead) * D);
        }
      }
      __syncthreads();
      conv_tile<D>(sg + OFF_RAW, reinterpret_cast<const float*>(sg + OFF_TAPS), sg + OFF_U, tid, 128, sg + OFF_UL);
      fence_proxy_async();
      tc_fence_before_sync();
      __syncthreads();
      tc_fence_after_sync();
      if (tid == 0) {  // Y = u W_h
        const uint32_t idesc = instr_desc(128, D, FMT_F16, MAJOR_K, MAJOR_MN);
        const uint64_t da = kview(sb + OFF_U, L::SLAB_U), db = mview(sb + OFF_WT, L::SLAB_W);
        for (int kk = 0; kk < D / 16; ++kk) mma_f16(tmem + COL_Y, dadv(da, 2 * L::SLAB_U * kk), dadv(db, 256 * kk), idesc, kk > 0);
        const uint64_t dal = kview(sb + OFF_UL, L::SLAB_U);  // (second term of u: the same features as the forward recompute)
        for (int kk = 0; kk < D / 16; ++kk) mma_f16(tmem + COL_Y, dadv(dal, 2 * L::SLAB_U * kk), dadv(db, 256 * kk), idesc, 1);
        mma_commit(sb + OFF_BAR);
      }
      wt.wait();
      // p = softmax(y), dy = p (dp - p . dp): this thread's row, two-term fp16 operand (rows past the end: zero)
      {
        float y[D];
        tmem_ld32(lane_base + COL_Y, y);
        tmem_ld32(lane_base + COL_Y + 32, y + 32);
        tmem_wait_ld();
        float m = -INFINITY, sum = 0.f, dot = 0.f;
#pragma unroll
        for (int i = 0; i < D; ++i) m = fmaxf(m, y[i]);
        const float mb = m * 1.4426950408889634f;
#pragma unroll
        for (int i = 0; i < D; ++i) {
          y[i] = ex2f(fmaf(y[i], 1.4426950408889634f, -mb));
          sum += y[i];
        }
        const float inv = 1.f / sum;
        const TG* dp = reinterpret_cast<const TG*>(stream ? a.d_kdot : a.d_qdot) + (((size_t)b * a.T + t) * a.H + h) * D;
#pragma unroll 1
        for (int pass = 0; pass < 2; ++pass) {
#pragma unroll
          for (int c0 = 0; c0 < D; c0 += 8) {
            float g8[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
            if (valid) load_row8(dp + c0, g8);
            if (pass == 0) {
#pragma unroll
              for (int i = 0; i < 8; ++i) dot = fmaf(y[c0 + i] * inv, g8[i], dot);
            } else {
              float dy[8], hi[8], lo[8];
#pragma unroll
              for (int i = 0; i < 8; ++i) dy[i] = valid ? y[c0 + i] * inv * (g8[i] - dot) : 0.f;
              const uint4 ph = pack8f16(dy);
              const __half2* h2 = reinterpret_cast<const __half2*>(&ph);
#pragma unroll
              for (int i = 0; i < 4; ++i) {
                const float2 f = __half22float2(h2[i]);
                hi[2 * i] = f.x; hi[2 * i + 1] = f.y;
              }
#pragma unroll
              for (int i = 0; i < 8; ++i) lo[i] = dy[i] - hi[i];
              *reinterpret_cast<uint4*>(sg + OFF_DY + toff(L::SLAB_U, tid, c0)) = ph;
              *reinterpret_cast<uint4*>(sg + OFF_DYL + toff(L::SLAB_U, tid, c0)) = pack8f16(lo);
            }
          }
        }
      }
      fence_proxy_async();
      tc_fence_before_sync();
      __syncthreads();
      tc_fence_after_sync();
      if (tid == 0) {
        // du = dy W_h^T (two-term dy) into Y's columns; dW_h += u^T dy
        const uint32_t id_du = instr_desc(128, D, FMT_F16, MAJOR_K, MAJOR_K);
        const uint64_t dh = kview(sb + OFF_DY, L::SLAB_U), dl = kview(sb + OFF_DYL, L::SLAB_U), dw = kview(sb + OFF_WT, L::SLAB_W);
        for (int kk = 0; kk < D / 16; ++kk) mma_f16(tmem + COL_Y, dadv(dh, 2 * L::SLAB_U * kk), dadv(dw, 2 * L::SLAB_W * kk), id_du, kk > 0);
        for (int kk = 0; kk < D / 16; ++kk) mma_f16(tmem + COL_Y, dadv(dl, 2 * L::SLAB_U * kk), dadv(dw, 2 * L::SLAB_W * kk), id_du, 1);
        const uint32_t id_dw = instr_desc(128, D, FMT_F16, MAJOR_MN, MAJOR_MN);
        // (both factors two-term: u_hi dy_hi + u_lo dy_hi + u_hi dy_lo; with few tokens in a call the weight gradient is
        // a sum of few products and the rounding of single 16-bit operands would show in its largest entries)
        const uint64_t ua = mview(sb + OFF_U, L::SLAB_U), ual = mview(sb + OFF_UL, L::SLAB_U);
        const uint64_t yb = mview(sb + OFF_DY, L::SLAB_U), ybl = mview(sb + OFF_DYL, L::SLAB_U);
        for (int kk = 0; kk < TT / 16; ++kk)
          mma_f16(tmem + COL_DW + 64 * (g & 1), dadv(ua, 256 * kk), dadv(yb, 256 * kk), id_dw, (stream > 0 || kk > 0) ? 1u : 0u);
        for (int kk = 0; kk < TT / 16; ++kk)
          mma_f16(tmem + COL_DW + 64 * (g & 1), dadv(ual, 256 * kk), dadv(yb, 256 * kk), id_dw, 1u);
        for (int kk = 0; kk < TT / 16; ++kk)
          mma_f16(tmem + COL_DW + 64 * (g & 1), dadv(ua, 256 * kk), dadv(ybl, 256 * kk), id_dw, 1u);
        mma_commit(sb + OFF_BAR);
      }
      wt.wait();
      {
        float du[D];
        tmem_ld32(lane_base + COL_Y, du);
        tmem_ld32(lane_base + COL_Y + 32, du + 32);
        tmem_wait_ld();
        if (stream == 0) {
          if (valid) {
            float* dst = a.du_q + (((size_t)b * a.T + t) * a.H + h) * D;
#pragma unroll
            for (int c0 = 0; c0 < D; c0 += 8) store_row8(dst + c0, du + c0);
          }
        } else {
#pragma unroll
          for (int i = 0; i < D; ++i) duk[i] += du[i];
        }
      }
      tc_fence_before_sync();
      __syncthreads();
      tc_fence_after_sync();
    }
    // dW of the last two heads (or the last one): row c of each accumulator is owned by thread c
    if (((g & 1) || g == G - 1) && warp < 2 && a.dW) {
#pragma unroll 1
      for (int gg = g & ~1; gg <= g; ++gg) {
        float r[32];
#pragma unroll 1
        for (int c0 = 0; c0 < D; c0 += 32) {
          tmem_ld32(lane_base + COL_DW + 64 * (gg & 1) + c0, r);
          tmem_wait_ld();
          float* dst = a.dW + ((size_t)(j * G + gg) * D + tid) * D + c0;
#pragma unroll
          for (int i = 0; i < 32; ++i) atomicAdd(dst + i, r[i]);
        }
      }
    }
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
  }
  if (valid) {
    float* dst = a.du_k + (((size_t)b * a.T + t) * a.Hkv + j) * D;
#pragma unroll
    for (int c0 = 0; c0 < D; c0 += 8) store_row8(dst + c0, duk + c0);
  }
  tc_fence_before_sync();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after_sync();
    tmem_dealloc(tmem, TMEM_COLS);
  }
}

constexpr uint32_t bwd_smem() {
  using L = Lay<64>;
  return L::TILE_W + 4 * L::TILE_U + 2048 + (L::RAW_BYTES + 15) / 16 * 16 + 64 * 16 + 64;
}

template <typename K>
static int raise_smem(K kernel, uint32_t bytes) {
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) == cudaSuccess ? LAWCAT_OK : LAWCAT_ERR_CUDA;
}

}  // namespace ctc

bool convmix_tc_fwd_supported(const lawcat_params& p) {
  return p.dtype == LAWCAT_BF16 && (p.d_k == 64 || p.d_k == 128) && p.conv_k <= ctc::HALO + 1 && p.B > 0 && p.T > 0;
}
bool convmix_tc_bwd_supported(const lawcat_params& p) {
  return p.dtype == LAWCAT_BF16 && p.d_k == 64 && p.phi == LAWCAT_PHI_SOFTMAX && p.conv_k <= ctc::HALO + 1 && p.B > 0 &&
         p.T > 0 && !p.mix_unshared;
}

static ctc::CArgs convmix_tc_args(const Ctx& c, const void* q, const void* k, const void* w_q, const void* w_k, const void* W,
                                  const void* cache_q, const void* cache_k) {
  const lawcat_params& p = *c.p;
  ctc::CArgs a{};
  a.q = (const bf16*)q; a.k = (const bf16*)k; a.w_q = (const bf16*)w_q; a.w_k = (const bf16*)w_k; a.W = (const bf16*)W;
  a.cache_q = (const bf16*)cache_q; a.cache_k = (const bf16*)cache_k;
  a.dev_status = c.dev_status;
  a.B = p.B; a.T = p.T; a.H = p.H; a.Hkv = p.H_kv; a.K = p.conv_k; a.phi = p.phi; a.unshared = p.mix_unshared;
  return a;
}

// qdot, kdot = softmax((conv x) W_h) for both streams; out_f32: fp32 outputs (scratch of a fused caller) instead of bf16
int launch_convmix_tc_fwd(const Ctx& c, const void* q, const void* k, const void* w_q, const void* w_k, const void* W,
                          const void* cache_q, const void* cache_k, void* qdot, void* kdot, bool out_f32) {
  using namespace ctc;
  const lawcat_params& p = *c.p;
  CArgs a = convmix_tc_args(c, q, k, w_q, w_k, W, cache_q, cache_k);
  a.qdot = qdot; a.kdot = kdot;
  static std::mutex mu;
  static bool done[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return LAWCAT_ERR_CUDA;
  {
    std::lock_guard<std::mutex> lk(mu);
    if (!done[dev]) {
      if (raise_smem(convmix_tc_fwd_kernel<64, bf16>, FwdMap<64, bf16>::BYTES) || raise_smem(convmix_tc_fwd_kernel<64, float>, FwdMap<64, float>::BYTES) ||
          raise_smem(convmix_tc_fwd_kernel<128, bf16>, FwdMap<128, bf16>::BYTES) || raise_smem(convmix_tc_fwd_kernel<128, float>, FwdMap<128, float>::BYTES))
        return LAWCAT_ERR_CUDA;
      done[dev] = true;
    }
  }
  const dim3 grid = tile_grid(p.B * p.H, p.T);
  LaunchScope _ls("convmix_tc_fwd", c.stream);
  if (p.d_k == 64) {
    if (out_f32) launch_behind(convmix_tc_fwd_kernel<64, float>, grid, dim3(fwd_threads<64, float>()), FwdMap<64, float>::BYTES, c.stream, a);
    else launch_behind(convmix_tc_fwd_kernel<64, bf16>, grid, dim3(fwd_threads<64, bf16>()), FwdMap<64, bf16>::BYTES, c.stream, a);
  } else {
    if (out_f32) launch_behind(convmix_tc_fwd_kernel<128, float>, grid, dim3(fwd_threads<128, float>()), FwdMap<128, float>::BYTES, c.stream, a);
    else launch_behind(convmix_tc_fwd_kernel<128, bf16>, grid, dim3(fwd_threads<128, bf16>()), FwdMap<128, bf16>::BYTES, c.stream, a);
  }
  LAWCAT_CHECK_LAUNCH();
  return LAWCAT_OK;
}

// du_q, du_k (fp32) and dW (atomic adds into the caller-zeroed array) from d_qdot, d_kdot
int launch_convmix_tc_bwd(const Ctx& c, const void* q, const void* k, const void* w_q, const void* w_k, const void* W,
                          const void* cache_q, const void* cache_k, const void* d_qdot, const void* d_kdot,
                          float* du_q, float* du_k, float* dW) {
  using namespace ctc;
  const lawcat_params& p = *c.p;
  CArgs a = convmix_tc_args(c, q, k, w_q, w_k, W, cache_q, cache_k);
  a.d_qdot = d_qdot; a.d_kdot = d_kdot; a.du_q = du_q; a.du_k = du_k; a.dW = dW;
  static std::mutex mu;
  static bool done[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return LAWCAT_ERR_CUDA;
  {
    std::lock_guard<std::mutex> lk(mu);
    if (!done[dev]) {
      if (raise_smem(convmix_tc_bwd_kernel, bwd_smem())) return LAWCAT_ERR_CUDA;
      done[dev] = true;
    }
  }
  const dim3 grid = tile_grid(p.B * p.H_kv, p.T);
  LaunchScope _ls("convmix_tc_bwd", c.stream);
  convmix_tc_bwd_kernel<<<grid, 128, bwd_smem(), c.stream>>>(a);
  LAWCAT_CHECK_LAUNCH();
  return LAWCAT_OK;
}

}  // namespace lawcat
