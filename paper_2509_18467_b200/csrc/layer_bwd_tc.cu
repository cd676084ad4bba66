// The attention part of the whole layer's backward (lawcat_layer_bwd; Section 5.1's distillation step) on the tensor cores,
// bf16 storage, d_k = d_v = 64 or 128, softmax feature map. The features qdot, kdot come in fp32 from the recomputed conv +
// mix; what goes out towards the mix is not their gradients but the products
//     wq = qdot * dqdot,   wk = kdot * dkdot   (elementwise)
// because that is all the softmax Jacobian needs (dy = w - p sum(w)) and all the gate gradient needs (dg_s = sum_{t>=s} wq_t -
// wk_t): the decay factors 2^{+-x} of the chunkwise form cancel in them and never have to be undone.
//
// With b_t the running sum of the log2-decays inside a chunk of C = 64 tokens, m = 31, x_t = b_t - b_m, bm = b_m, ft = b_C - b_m:
//   qs_t = qdot_t 2^{x_t},  ks_i = kdot_i 2^{-x_i},  S16 = 2^bm S (S the state in front of the chunk, z its normalizer column)
//   forward sweep   P = mask(qs ks^T)    num | den = P [v|1] + qs [S16|z16]    W <- S16 + ks^T [v|1]   (next state = 2^ft W)
//                   inv_t = 1 / den_t, delta_t = dO_t . o_t; the operand S16 of every chunk is kept for the reverse sweep
//   reverse sweep   qn_t = qs_t inv_t      P' = mask(qn ks^T)      E = mask(dO v^T - delta_t)
//                   dQ = E ks + dO S16^T - delta z16             wq = qn * dQ
//                   dK = E^T qn + v R16^T + r16                  wk = ks * dK      (R16 = 2^ft R, R the adjoint of the state
//                   dV = P'^T dO + ks R16                                           behind the chunk, r its normalizer column)
//                   W' <- R16 + qn^T dO  (adjoint in front of the chunk = 2^bm W')   r likewise with -delta
// Dividing by den is folded into qn and into the row terms, so dO and v enter every product unrounded (both are exact in 16
// bits); qn, ks, S16, R16, P' and E are two-term 16-bit pairs hi + lo (hi hi + lo hi + hi lo: about 21 bits). Powers of two keep
// the pairs in the fp16 range and away from its subnormals: 2^kap on ks and S16 (per chunk, from a bound on the state), 2^al on
// inv (per chunk, from its largest inv and the largest adjoint entry), 2^sc on dO (per head, from its largest |dO| and a bound on
// E). Chunks whose decay exponents leave +-8, or whose v is beyond the fp16 range, use bf16 pairs.
//
// One thread block walks one (batch, query head), lock-step: every phase of a chunk by all threads, products by one thread
// (tcgen05.mma, fp32 accumulators in tensor memory), bounded waits on mbarriers. What bounds it is that chain of phases:
// instruction issue in the operand and epilogue passes, the products second. Head width 64: two blocks per SM (<= 113 KB, 256
// tensor memory columns); 128: one block of 512 threads.
#include <cuda.h>
#include <cuda_fp16.h>

#include <mutex>
#include <type_traits>

#include "common.cuh"
#include "octet_tile.cuh"
#include "tc_common.cuh"

namespace lawcat {
namespace lbt {

using namespace tc;
using namespace ctc;

constexpr int C = 64, MID = 31;
constexpr float RMAX_F16 = 8.f, VMAX_F16 = 65504.f;
constexpr int QSC = 4;       // power of two on qs in the forward sweep
constexpr int KAP_MAX = 4;   // largest power of two on ks and S16 (ks <= 2^8 in fp16 chunks)

struct Args {
  const float *qd, *kd;                 // [B,T,H,D] features
  const bf16 *v, *gate, *dO;
  const float *S0, *z0;
  float *wq, *wk;                       // [B,T,H,D]
  float* dvh;                           // [B,T,H,D] per-head dv, reduced over the heads of a group afterwards
  bf16* dgate;
  float *inv, *delta;                   // [B,T,H]
  float2* domax;                        // [B*H] of the head: largest |dO|, and a bound on |dO . v_i - delta|
  float* z16;                           // [B*H][chunks][D]
  int* meta;                            // [B*H][chunks][2]: kap, operand format
  uint8_t* s16;                         // [B*H][chunks][2 * D * D * 2] operand tiles, hi then lo
  float* wmax;                          // [B*H] largest |wq|, |wk| of the head
  float* dW;                            // [H,D,D] weight gradient, accumulated by the mix backward: zeroed by the sweep
  float* du_k;                          // [B,T,Hkv,D], zeroed as well where several blocks of the mix backward add to it (else null)
  int* dev_status;
  int B, T, H, Hkv, gate_dim, gate_mode, normalize;
  float inv_tau, eps;
};

struct Maps {  // tensor maps [B,T,heads,D]: whole rows of 64 tokens for the prefetch, 32 fp32 channels x 64 tokens for the stores
  CUtensorMap qd, kd, v, dO, wq, wk, dvh;
};

template <int D>
struct Cfg {
  static constexpr int THREADS = D == 128 ? 512 : 256, OCT = D / 8, NCG = THREADS / 128;  // NCG: column groups of row threads
  static constexpr uint32_t SL_T = C * 16 + 16;  // slab stride of token tiles written eight lanes to a row (padded: the slabs
                                                 // then start in different banks)
  static constexpr uint32_t SL_U = C * 16;       // ... of token tiles written a lane to a row
  static constexpr uint32_t SL_C = D * 16;       // ... of tiles with D rows
  static constexpr uint32_t T_TOK = OCT * SL_T, T_P = 8 * SL_U, T_C = OCT * SL_C;
  // forward sweep
  static constexpr uint32_t F_QS = 0, F_KS = F_QS + 2 * T_TOK, F_V = F_KS + 2 * T_TOK, F_PM = F_V + (OCT + 2) * SL_T;
  static constexpr uint32_t F_S = F_PM + 2 * T_P, T_SZ = (OCT + 2) * SL_C, F_VEC = F_S + 2 * T_SZ;
  static constexpr uint32_t F_BYTES = F_VEC + 4 * D * 4 + NCG * C * 4 + 64;
  static constexpr uint32_t F_X = F_S;           // exponents, fp32 [C][D]: dead before the state operand is written
  // reverse sweep
  static constexpr uint32_t R_QS = 0, R_KS = R_QS + 2 * T_TOK, R_V = R_KS + 2 * T_TOK, R_DO = R_V + T_TOK,
                            R_PM = (R_DO + T_TOK + 1023) / 1024 * 1024;  // (result tiles that lie here and behind are swizzled)
  static constexpr uint32_t R_E = R_PM + 2 * T_P, R_S = R_E + 2 * T_P, R_VEC = R_S + 2 * T_C;
  static constexpr uint32_t R_BYTES = R_VEC + 8 * D * 4 + 2 * C * 4 + (THREADS / 32) * D * 4 + 96;
  static constexpr uint32_t R_X = R_S;
  // fp32 [C][D] result tiles over operands that are dead by then
  static constexpr uint32_t R_WQ = R_S, R_WK = D == 128 ? R_S + C * D * 4 : R_PM, R_DV = D == 128 ? R_PM : R_E, R_DG = R_QS;
  static_assert(C * D * 4 <= 2 * T_SZ && C * D * 4 <= 2 * T_TOK && 2 * T_P >= C * 64 * 4, "aliases");
  static_assert(R_WQ % 1024 == 0 && R_WK % 1024 == 0 && R_DV % 1024 == 0, "the copy engine's swizzle goes by the address");
  static_assert(R_BYTES <= (D == 128 ? 232448 : 115000) && F_BYTES <= (D == 128 ? 232448 : 115000), "shared memory budget");
  // tensor memory
  static constexpr uint32_t F_ST = 0, F_O = D + 16, F_P = 2 * (D + 16), COLS = D == 128 ? 512 : 256;
  static constexpr uint32_t R_R = 0, R_DQ = D, R_DK = 2 * D, R_DVC = 3 * D, R_P = R_DQ, R_EP = R_DQ + 64;
};

__device__ __forceinline__ float pow2i(int e) { return __int_as_float((min(max(e, -126), 127) + 127) << 23); }
// smallest e with |x| < 2^e (x > 0)
__device__ __forceinline__ int exp_above(float x) { return ((__float_as_int(x) >> 23) & 0xff) - 126; }
// piece pc (16 bytes) of row r of an fp32 [C][D] tile: slabs of 32 columns, 128-byte-swizzled as the copy engine stores them, so that
// lanes that own rows spread over the banks
__device__ __forceinline__ uint32_t foff(int r, int pc) { return (uint32_t)((pc >> 3) * (C * 128)) + sw128(r, pc & 7); }

// A chunk's gate entries as they lie in memory, two octets per thread (gate_dim = 1: the token's entry as fp32 bits), fetched
// while the chunk in front is computed.
template <int D>
struct Gates {
  uint4 r[2];
  __device__ __forceinline__ void load(const Args& a, int b, int h, int t0, int tid) {
    using F = Cfg<D>;
    static_assert(C * F::OCT == 2 * F::THREADS, "two octets per thread");
#pragma unroll
    for (int it = 0; it < 2; ++it) {
      const int idx = tid + it * F::THREADS, o = idx % F::OCT, t = t0 + idx / F::OCT;
      r[it] = make_uint4(0u, 0u, 0u, 0u);
      if (t0 >= 0 && t < a.T) {
        const size_t gi = ((size_t)b * a.T + t) * a.H + h;
        if (a.gate_dim == 1) r[it].x = __float_as_uint(__bfloat162float(a.gate[gi]));
        else r[it] = *reinterpret_cast<const uint4*>(a.gate + gi * D + o * 8);
      }
    }
  }
};

// Log-decays of a chunk scanned outwards from the middle token: exponents x into s_x (fp32, rows of D), bm and ft per channel,
// the largest |x| into *rmax (cleared by the caller behind a barrier). Ends with a barrier; the caller has one between the
// last readers of s_x and this call.
template <int D>
__device__ __forceinline__ void gate_pass(const Args& a, const Gates<D>& raw, int nvalid, float* s_x, float* s_bm, float* s_ft,
                                          int* rmax, int tid) {
  using F = Cfg<D>;
  const float L2E = 1.4426950408889634f;
#pragma unroll
  for (int it = 0; it < 2; ++it) {
    const int idx = tid + it * F::THREADS, o = idx % F::OCT, r = idx / F::OCT;
    float g[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    if (r < nvalid) {
      if (a.gate_dim == 1) {
        const float av = __uint_as_float(raw.r[it].x);
        const float gv = a.gate_mode == LAWCAT_GATE_LOGDECAY ? av * L2E : log2_sigmoid(av) * a.inv_tau;
#pragma unroll
        for (int i = 0; i < 8; ++i) g[i] = gv;
      } else {
        unpack8b(raw.r[it], g);
        if (a.gate_mode == LAWCAT_GATE_LOGDECAY) {
#pragma unroll
          for (int i = 0; i < 8; ++i) g[i] *= L2E;
        } else {
#pragma unroll
          for (int i = 0; i < 8; ++i) g[i] = log2_sigmoid(g[i]) * a.inv_tau;
        }
      }
    }
    store_row8(s_x + r * D + o * 8, g);
  }
  __syncthreads();
  if (tid < 2 * D) {
    const int c = tid & (D - 1), gh = tid / D;
    float g[32], acc = 0.f;
#pragma unroll
    for (int i = 0; i < 32; ++i) g[i] = s_x[(gh * 32 + i) * D + c];
    if (gh) {
#pragma unroll
      for (int i = 0; i < 32; ++i) {
        acc += g[i];
        s_x[(32 + i) * D + c] = fmaxf(acc, -120.f);
      }
      s_ft[c] = acc;
    } else {
      s_x[MID * D + c] = 0.f;
#pragma unroll
      for (int i = MID - 1; i >= 0; --i) {
        acc += g[i + 1];
        s_x[i * D + c] = fminf(-acc, 120.f);
      }
      s_bm[c] = acc + g[0];
    }
    if (-acc > 120.f && a.dev_status) atomicMax(a.dev_status, (int)LAWCAT_ERR_NUMERIC);
    const float am = warp_max(-acc);
    if ((tid & 31) == 0) atomicMax(rmax, __float_as_int(am));
  }
  __syncthreads();
}

// One chunk's rows towards L2, by one thread and four instructions while a batch of products is under way: the chunk that follows
// travels while this one is computed. (Line by line, by the warps that wait, it took them 5k cycles a chunk at width 128, longer than
// the products.)
__device__ __forceinline__ void prefetch_chunk(const Maps& m, int b, int h, int j, int t0) {
  tma_prefetch_4d(&m.qd, 0, h, t0, b);
  tma_prefetch_4d(&m.kd, 0, h, t0, b);
  tma_prefetch_4d(&m.v, 0, j, t0, b);
  tma_prefetch_4d(&m.dO, 0, h, t0, b);
}

// A chunk's rows as they lie in memory, two octets per thread, loaded before the gate pass so that they arrive behind it.
template <int D, bool REV>
struct Rows {
  float4 q[2][2], k[2][2];
  uint4 v[2], g[2];
  __device__ __forceinline__ void load(const Args& a, size_t row0, int h, int j, int nvalid, int tid) {
    using F = Cfg<D>;
#pragma unroll
    for (int it = 0; it < 2; ++it) {
      const int idx = tid + it * F::THREADS, o = idx % F::OCT, r = idx / F::OCT;
      const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
      q[it][0] = q[it][1] = k[it][0] = k[it][1] = z;
      v[it] = g[it] = make_uint4(0u, 0u, 0u, 0u);
      if (r < nvalid) {
        const size_t tq = ((row0 + r) * a.H + h) * D + o * 8;
        load_octet(a.qd + tq, q[it]);
        load_octet(a.kd + tq, k[it]);
        v[it] = *reinterpret_cast<const uint4*>(a.v + ((row0 + r) * a.Hkv + j) * D + o * 8);
        if (REV) g[it] = *reinterpret_cast<const uint4*>(a.dO + tq);
      }
    }
  }
  static __device__ __forceinline__ void f8(const float4 (&x)[2], float* f) {
    f[0] = x[0].x; f[1] = x[0].y; f[2] = x[0].z; f[3] = x[0].w; f[4] = x[1].x; f[5] = x[1].y; f[6] = x[1].z; f[7] = x[1].w;
  }
};

// products on two-term operands, issued by one lane: D (+)= A B with A = ah + al, B = bh + bl (a missing low part is 0). (The
// issuing lane is an elected one of a uniform warp: reverse sweep of 8 x 1024 tokens of 32 heads of 64 255 -> 244 us. Rolled: the 128
// products of a chunk of the reverse sweep at width 128, unrolled, cost 359 us instead of 350.)
struct Mma {
  uint32_t tmem;
  __device__ __forceinline__ void chain(uint32_t col, uint64_t da, uint32_t as, uint64_t db, uint32_t bs, int ks, uint32_t id, bool acc) const {
#pragma unroll 1
    for (int k = 0; k < ks; ++k) mma_f16(tmem + col, dadv(da, as * k), dadv(db, bs * k), id, (acc || k > 0) ? 1u : 0u);
  }
  __device__ __forceinline__ void split(uint32_t col, uint64_t ah, uint64_t al, uint32_t as, uint64_t bh, uint64_t bl, uint32_t bs,
                                        int ks, uint32_t id, bool acc) const {
    chain(col, ah, as, bh, bs, ks, id, acc);
    if (al) chain(col, al, as, bh, bs, ks, id, true);
    if (bl) chain(col, ah, as, bl, bs, ks, id, true);
  }
};

// ------------------------------------------------------------------------------------------------ forward sweep
template <int D>
__global__ void __launch_bounds__(Cfg<D>::THREADS, D == 128 ? 1 : 2) sweep_kernel(const Args a, const __grid_constant__ Maps maps) {
  using F = Cfg<D>;
  constexpr int NV = D + 16;
  extern __shared__ __align__(128) uint8_t sg[];
  const uint32_t sb = smem_u32(sg);
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;  // (warp: uniform to the compiler)
  float* const s_x = reinterpret_cast<float*>(sg + F::F_X);
  float* const s_bm = reinterpret_cast<float*>(sg + F::F_VEC);
  float *const s_ft = s_bm + D, *const s_pe = s_ft + D;  // s_pe: ft of the chunk in front (its state is still 2^-ft short)
  float* const s_row = s_pe + 2 * D;                     // [NCG][C]
  volatile int* const s_fl = reinterpret_cast<volatile int*>(s_row + F::NCG * C);  // tmem base, abort, rmax, smax, vmax, domax, dlmax
  const uint32_t bar = smem_u32(const_cast<int*>(s_fl)) + 32, bar_p = bar + 8;
  const int bh = blockIdx.x, h = bh % a.H, b = bh / a.H, G = a.H / a.Hkv, j = h / G;
  const int nch = (a.T + C - 1) / C;
  if (tid == 0) {
    mbar_init(bar, 1);
    mbar_init(bar_p, 1);
    mbar_fence_init();
    for (int i = 1; i < 7; ++i) s_fl[i] = 0;
  }
  if (warp == 0) {
    tmem_alloc(smem_u32(const_cast<int*>(s_fl)), F::COLS);
    tmem_relinquish();
  }
  asm volatile("griddepcontrol.wait;" ::: "memory");  // (each kernel of the step is launched behind the one in front)
  // dW is zeroed here (every block a part) and not by a memset node of its own, which costs microseconds
  for (int i = blockIdx.x * F::THREADS + tid; i < a.H * D * D / 4; i += gridDim.x * F::THREADS)
    reinterpret_cast<float4*>(a.dW)[i] = make_float4(0.f, 0.f, 0.f, 0.f);
  if (a.du_k) {
    const size_t n4 = (size_t)a.B * a.T * a.Hkv * (D / 4);
    for (size_t i = (size_t)blockIdx.x * F::THREADS + tid; i < n4; i += (size_t)gridDim.x * F::THREADS)
      reinterpret_cast<float4*>(a.du_k)[i] = make_float4(0.f, 0.f, 0.f, 0.f);
  }
  // the two extra slabs of [v | 1] (column D: the 1) and of the state operand (column D: z; the rest zero)
  for (int i = tid; i < 2 * C; i += F::THREADS)
    *reinterpret_cast<uint4*>(sg + F::F_V + toff(F::SL_T, i & (C - 1), D + 8 * (i >> 6))) = make_uint4(0u, 0u, 0u, 0u);
  for (int i = tid; i < D; i += F::THREADS) s_pe[i] = 0.f;
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const Mma mm{(uint32_t)s_fl[0]};
  const uint32_t lane_base = mm.tmem + ((uint32_t)((warp & 3) * 32) << 16);
  const int row = (warp & 3) * 32 + lane, cg = warp >> 2;  // TMEM lane, column group
  const bool tok_thr = row < C, st_thr = row < D;          // owns a token row / a state row
  Waiter wt{bar, 0u, s_fl + 1, a.dev_status}, wp{bar_p, 0u, s_fl + 1, a.dev_status};
  constexpr int SW = D / F::NCG, TW = 64 / F::NCG;         // columns per thread of a state row, of a score row
  auto publish = [&]() {
    fence_proxy_async();
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
  };
  float smx = 0.f;
  if (st_thr) {
    float s[8];
#pragma unroll 1
    for (int c0 = cg * SW; c0 < (cg + 1) * SW; c0 += 8) {
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        s[i] = a.S0 ? a.S0[((size_t)bh * D + row) * D + c0 + i] : 0.f;
        smx = fmaxf(smx, fabsf(s[i]));
      }
      tmem_st8(lane_base + F::F_ST + c0, s);
    }
    if (cg == 0) {
#pragma unroll
      for (int i = 0; i < 8; ++i) s[i] = 0.f;
      tmem_st8(lane_base + F::F_ST + D + 8, s);
      s[0] = a.z0 ? a.z0[(size_t)bh * D + row] : 0.f;
      smx = fmaxf(smx, fabsf(s[0]));
      tmem_st8(lane_base + F::F_ST + D, s);
    }
    tmem_wait_st();
  }
  if (!(smx < 1.0e30f)) smx = 1.0e30f;
  smx = warp_max(smx);
  if (lane == 0) atomicMax(const_cast<int*>(&s_fl[3]), __float_as_int(smx));
  __syncthreads();
  float sbound = __int_as_float(s_fl[3]), domax = 0.f, dlmax = 0.f, vhead = 0.f;  // (largest |dO|, |delta|, |v| so far)
  int kap_prev = 0;
  Gates<D> gates;
  gates.load(a, b, h, 0, tid);
  auto KV = [&](uint32_t off, uint32_t slab) -> uint64_t { return kview(sb + off, slab); };
  auto MV = [&](uint32_t off, uint32_t slab) -> uint64_t { return mview(sb + off, slab); };

  for (int n = 0; n < nch; ++n) {
    const int t0 = n * C, nvalid = min(C, a.T - t0);
    const size_t row0 = (size_t)b * a.T + t0;
    Rows<D, false> rows;
    rows.load(a, row0, h, j, nvalid, tid);
    gate_pass<D>(a, gates, nvalid, s_x, s_bm, s_ft, const_cast<int*>(&s_fl[2]), tid);
    bool f16 = __int_as_float(s_fl[2]) <= RMAX_F16;
    const int kap = max(-100, min(KAP_MAX, 14 - exp_above(fmaxf(sbound, 1e-30f))));
    const float ksc = pow2i(kap);
    // ---- operands
    auto operands = [&](bool f16) {
      float vmax = 0.f;
#pragma unroll
      for (int it = 0; it < 2; ++it) {
        const int idx = tid + it * F::THREADS, o = idx % F::OCT, r = idx / F::OCT;
        float q[8], k[8], vv[8], x[8];
        rows.f8(rows.q[it], q);
        rows.f8(rows.k[it], k);
        unpack8b(rows.v[it], vv);
        load_row8(s_x + r * D + o * 8, x);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          q[i] *= ex2f(x[i]) * (float)(1 << QSC);
          k[i] *= ex2f(-x[i]) * ksc;
          vmax = fmaxf(vmax, fabsf(vv[i]));
        }
        uint4 hi, lo;
        const uint32_t at = toff(F::SL_T, r, o * 8);
        split8h(q, f16, hi, lo);
        *reinterpret_cast<uint4*>(sg + F::F_QS + at) = hi;
        *reinterpret_cast<uint4*>(sg + F::F_QS + F::T_TOK + at) = lo;
        split8h(k, f16, hi, lo);
        *reinterpret_cast<uint4*>(sg + F::F_KS + at) = hi;
        *reinterpret_cast<uint4*>(sg + F::F_KS + F::T_TOK + at) = lo;
        *reinterpret_cast<uint4*>(sg + F::F_V + at) = pack8h(vv, f16);
        if (o == 0) {
          const float one[8] = {1.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
          *reinterpret_cast<uint4*>(sg + F::F_V + toff(F::SL_T, r, D)) = pack8h(one, f16);
        }
      }
      vmax = warp_max(vmax);
      if (lane == 0) atomicMax(const_cast<int*>(&s_fl[4]), __float_as_int(vmax < 1.0e30f ? vmax : 1.0e30f));
    };
    operands(f16);
    __syncthreads();  // (the exponents have been read: the state operand may overwrite them)
    if (f16 && __int_as_float(s_fl[4]) > VMAX_F16) {  // v is beyond the fp16 range: once more, in bf16
      f16 = false;
      rows.load(a, row0, h, j, nvalid, tid);
      operands(false);
      __syncthreads();
    }
    const int fmt = f16 ? FMT_F16 : FMT_BF16;
    // ---- state pass: W = 2^(bm + ft of the chunk in front) S, kept in tensor memory and as the two-term operand, scaled 2^kap
    smx = 0.f;
    if (st_thr) {
      const float f = ex2f(fmaxf(s_bm[row] + s_pe[row], -126.f)) * pow2i(kap - kap_prev);
      static_assert(SW == 32, "one wide load");
      float y[32], s[8];
      uint4 hi, lo;
      tmem_ld32(lane_base + F::F_ST + cg * SW, y);
      tmem_wait_ld();
#pragma unroll
      for (int i8 = 0; i8 < 32; i8 += 8) {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          y[i8 + i] *= f;
          smx = fmaxf(smx, fabsf(y[i8 + i]));
        }
        split8h(y + i8, f16, hi, lo);
        *reinterpret_cast<uint4*>(sg + F::F_S + toff(F::SL_C, row, cg * SW + i8)) = hi;
        *reinterpret_cast<uint4*>(sg + F::F_S + F::T_SZ + toff(F::SL_C, row, cg * SW + i8)) = lo;
      }
      tmem_st32(lane_base + F::F_ST + cg * SW, y);
      if (cg == F::NCG - 1) {
        tmem_ld8(lane_base + F::F_ST + D, s);
        tmem_wait_ld();
        s[0] *= f;
        smx = fmaxf(smx, fabsf(s[0]));
#pragma unroll
        for (int i = 1; i < 8; ++i) s[i] = 0.f;
        split8h(s, f16, hi, lo);
        *reinterpret_cast<uint4*>(sg + F::F_S + toff(F::SL_C, row, D)) = hi;
        *reinterpret_cast<uint4*>(sg + F::F_S + F::T_SZ + toff(F::SL_C, row, D)) = lo;
        *reinterpret_cast<uint4*>(sg + F::F_S + toff(F::SL_C, row, D + 8)) = make_uint4(0u, 0u, 0u, 0u);
        *reinterpret_cast<uint4*>(sg + F::F_S + F::T_SZ + toff(F::SL_C, row, D + 8)) = make_uint4(0u, 0u, 0u, 0u);
        tmem_st8(lane_base + F::F_ST + D, s);
        a.z16[((size_t)bh * nch + n) * D + row] = s[0];
      }
      tmem_wait_st();
    }
    smx = warp_max(smx);
    if (lane == 0) atomicMax(const_cast<int*>(&s_fl[3]), __float_as_int(smx < 1.0e30f ? smx : 1.0e30f));
    publish();
    if (tid == 0) {
      uint8_t* dst = a.s16 + ((size_t)bh * nch + n) * (2 * F::T_C);
      asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst), "r"(sb + F::F_S), "r"(F::T_C) : "memory");
      asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst + F::T_C), "r"(sb + F::F_S + F::T_SZ), "r"(F::T_C) : "memory");
      tma_store_commit();
      a.meta[((size_t)bh * nch + n) * 2] = kap;
      a.meta[((size_t)bh * nch + n) * 2 + 1] = fmt;
    }
    if (warp == 0 && elect_one()) {
      mm.split(F::F_P, KV(F::F_QS, F::SL_T), KV(F::F_QS + F::T_TOK, F::SL_T), 2 * F::SL_T, KV(F::F_KS, F::SL_T),
               KV(F::F_KS + F::T_TOK, F::SL_T), 2 * F::SL_T, D / 16, instr_desc(128, C, fmt, MAJOR_K, MAJOR_K), false);
      mma_commit(bar_p);
      mm.split(F::F_O, KV(F::F_QS, F::SL_T), KV(F::F_QS + F::T_TOK, F::SL_T), 2 * F::SL_T, MV(F::F_S, F::SL_C),
               MV(F::F_S + F::T_SZ, F::SL_C), 256, D / 16, instr_desc(128, NV, fmt, MAJOR_K, MAJOR_MN), false);
      // (the state in tensor memory is 2^kap-scaled like ks)
      mm.split(F::F_ST, MV(F::F_KS, F::SL_T), MV(F::F_KS + F::T_TOK, F::SL_T), 256, MV(F::F_V, F::SL_T), 0, 256, C / 16,
               instr_desc(128, NV, fmt, MAJOR_MN, MAJOR_MN), true);
    }
    gates.load(a, b, h, t0 + C, tid);  // (early: these rows are not prefetched)
    if (tid == 32 && n + 1 < nch) prefetch_chunk(maps, b, h, j, t0 + C);
    wp.wait();  // (the scores alone: the mask runs behind the read-out and the state update)
    // ---- mask
    if (tok_thr) {
      float s[16];
      uint4 hi, lo;
#pragma unroll 1
      for (int c0 = cg * TW; c0 < (cg + 1) * TW; c0 += 16) {
        tmem_ld16(lane_base + F::F_P + c0, s);
        tmem_wait_ld();
#pragma unroll
        for (int i8 = 0; i8 < 16; i8 += 8) {
#pragma unroll
          for (int i = 0; i < 8; ++i) s[i8 + i] = c0 + i8 + i <= row ? s[i8 + i] : 0.f;
          split8h(s + i8, f16, hi, lo);
          *reinterpret_cast<uint4*>(sg + F::F_PM + toff(F::SL_U, row, c0 + i8)) = hi;
          *reinterpret_cast<uint4*>(sg + F::F_PM + F::T_P + toff(F::SL_U, row, c0 + i8)) = lo;
        }
      }
    }
    for (int i = tid; i < D; i += F::THREADS) s_pe[i] = s_ft[i];
    publish();
    if (warp == 0 && elect_one()) {
      mm.split(F::F_O, KV(F::F_PM, F::SL_U), KV(F::F_PM + F::T_P, F::SL_U), 2 * F::SL_U, MV(F::F_V, F::SL_T), 0, 256, C / 16,
               instr_desc(128, NV, fmt, MAJOR_K, MAJOR_MN), true);
      mma_commit(bar);
    }
    // |next state| <= |2^bm state| + 64 max|v|: every key enters with a factor <= 1
    const float vm = __int_as_float(s_fl[4]), sm = __int_as_float(s_fl[3]) * pow2i(-kap);
    wt.wait();
    // ---- 1 / den and dO . o of the chunk's rows
    float inv = 1.f, dot = 0.f;
    if (tok_thr) {
      const float den = tmem_ld1(lane_base + F::F_O + D);
      tmem_wait_ld();
      const float osc = pow2i(-(QSC + kap));
      inv = a.normalize ? 1.f / fmaf(den, osc, a.eps) : 1.f;
      const float oi = inv * osc;
      const bf16* g = a.dO + ((row0 + min(row, nvalid - 1)) * a.H + h) * D;
      float s[32];
      uint4 gr[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) gr[i] = *reinterpret_cast<const uint4*>(g + cg * SW + 8 * i);
      tmem_ld32(lane_base + F::F_O + cg * SW, s);
      tmem_wait_ld();
#pragma unroll
      for (int i8 = 0; i8 < 4; ++i8) {
        float gv[8];
        unpack8b(gr[i8], gv);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          dot = fmaf(gv[i], s[8 * i8 + i] * oi, dot);
          domax = fmaxf(domax, fabsf(gv[i]));
        }
      }
      s_row[cg * C + row] = dot;
    }
    if (tid == 0) tma_store_wait_read();  // (the state operand has left: the next chunk's exponents may overwrite it)
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    if (tid == 0) s_fl[2] = s_fl[3] = s_fl[4] = 0;
    if (tok_thr && cg == 0 && row < nvalid) {
      float d = 0.f;
#pragma unroll
      for (int i = 0; i < F::NCG; ++i) d += s_row[i * C + row];
      const size_t th = (row0 + row) * a.H + h;
      a.inv[th] = inv;
      a.delta[th] = a.normalize ? d : 0.f;
      if (a.normalize) dlmax = fmaxf(dlmax, fabsf(d));
    }
    sbound = sm + 64.f * fmaxf(vm, 1.f);
    vhead = fmaxf(vhead, vm);
    kap_prev = kap;
    __syncthreads();
  }
  domax = warp_max(domax);
  if (lane == 0) atomicMax(const_cast<int*>(&s_fl[5]), __float_as_int(domax < 1.0e30f ? domax : 1.0e30f));
  dlmax = warp_max(dlmax);
  if (lane == 0) atomicMax(const_cast<int*>(&s_fl[6]), __float_as_int(dlmax < 1.0e30f ? dlmax : 1.0e30f));
  tc_fence_before_sync();
  __syncthreads();
  if (tid == 0) {
    domax = __int_as_float(s_fl[5]);
    a.domax[bh] = make_float2(domax, (float)D * domax * vhead + __int_as_float(s_fl[6]));
    tma_store_wait_all();
  }
  if (warp == 0) {
    tc_fence_after_sync();
    tmem_dealloc(mm.tmem, F::COLS);
  }
}

// ------------------------------------------------------------------------------------------------ reverse sweep
template <int D>
__global__ void __launch_bounds__(Cfg<D>::THREADS, D == 128 ? 1 : 2) reverse_kernel(const Args a, const __grid_constant__ Maps maps) {
  using F = Cfg<D>;
  constexpr int NW = F::THREADS / 32;
  extern __shared__ __align__(1024) uint8_t sg[];
  const uint32_t sb = smem_u32(sg);
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;  // (warp: uniform to the compiler)
  float* const s_x = reinterpret_cast<float*>(sg + F::R_X);
  float* const s_bm = reinterpret_cast<float*>(sg + F::R_VEC);
  float *const s_ft = s_bm + D, *const s_pe = s_ft + D;  // s_pe: bm of the chunk behind (its adjoint is still 2^-bm short)
  float *const s_z = s_pe + D, *const s_r16 = s_z + D, *const s_r = s_r16 + D, *const s_car = s_r + D;
  float *const s_tot = s_car + D;                        // (unused tail of D floats keeps the row scalars aligned)
  float *const s_inv = s_tot + D, *const s_dl = s_inv + C;
  float* const s_rp = s_dl + C;                          // [NW][D] partial sums of r
  volatile int* const s_fl = reinterpret_cast<volatile int*>(s_rp + NW * D);  // tmem base, abort, rmax, imax, Rmax, wmax
  const uint32_t bar = smem_u32(const_cast<int*>(s_fl)) + 32, bar_s = bar + 8;
  const int bh = blockIdx.x, h = bh % a.H, b = bh / a.H, G = a.H / a.Hkv, j = h / G;
  const int nch = (a.T + C - 1) / C;
  if ((sb & 1023u) != 0) {  // (the swizzled result tiles need a 1024-byte aligned base)
    if (tid == 0 && a.dev_status) atomicMax(a.dev_status, (int)LAWCAT_ERR_CUDA);
    return;
  }
  if (tid == 0) {
    mbar_init(bar, 1);
    mbar_init(bar_s, 1);
    mbar_fence_init();
    for (int i = 1; i < 6; ++i) s_fl[i] = 0;
  }
  if (warp == 0) {
    tmem_alloc(smem_u32(const_cast<int*>(s_fl)), F::COLS);
    tmem_relinquish();
  }
  for (int i = tid; i < D; i += F::THREADS) s_pe[i] = s_r[i] = s_car[i] = 0.f;
  asm volatile("griddepcontrol.wait;" ::: "memory");
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const Mma mm{(uint32_t)s_fl[0]};
  const uint32_t lane_base = mm.tmem + ((uint32_t)((warp & 3) * 32) << 16);
  const int row = (warp & 3) * 32 + lane, cg = warp >> 2;
  const bool tok_thr = row < C, st_thr = row < D;
  Waiter wt{bar, 0u, s_fl + 1, a.dev_status}, ws{bar_s, 0u, s_fl + 1, a.dev_status};
  constexpr int SW = D / F::NCG, TW = 64 / F::NCG;
  auto publish = [&]() {
    fence_proxy_async();
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
  };
  auto KV = [&](uint32_t off, uint32_t slab) -> uint64_t { return kview(sb + off, slab); };
  auto MV = [&](uint32_t off, uint32_t slab) -> uint64_t { return mview(sb + off, slab); };
  if (st_thr) {  // the adjoint starts at zero
    float s[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll 1
    for (int c0 = cg * SW; c0 < (cg + 1) * SW; c0 += 8) tmem_st8(lane_base + F::R_R + c0, s);
    tmem_wait_st();
  }
  // 2^sc: the largest |dO| of the head becomes 2^4 .. 2^5 (every gradient is linear in dO), or less where |v| is so large (from
  // about 16 on for d = 128) that an entry of E could leave the fp16 range otherwise
  const float2 dmx = a.domax[bh];
  const int sc = min(5 - exp_above(fmaxf(dmx.x, 1e-30f)), 16 - exp_above(fmaxf(1.001f * dmx.y, 1e-30f)));
  const float osc = pow2i(sc);
  int al_prev = 0;
  float wmax = 0.f;
  int copied = -1;  // (first thread) the last copy of a state operand that was started
  // what the next chunk's first passes need, fetched while the chunk behind it is computed
  Gates<D> gates;
  int2 nx_meta = make_int2(0, 0);
  float nx_inv = 0.f, nx_dl = 0.f, nx_z = 0.f;
  auto fetch_next = [&](int m) {
    if (m < 0) return;
    gates.load(a, b, h, m * C, tid);
    nx_meta = *reinterpret_cast<const int2*>(a.meta + ((size_t)bh * nch + m) * 2);
    nx_inv = nx_dl = 0.f;
    if (tid < C && m * C + tid < a.T) {
      const size_t th = ((size_t)b * a.T + m * C + tid) * a.H + h;
      nx_inv = a.inv[th];
      nx_dl = a.delta[th];
    }
    if (tid >= C && tid < C + D) nx_z = a.z16[((size_t)bh * nch + m) * D + tid - C];
  };
  fetch_next(nch - 1);

  for (int n = nch - 1; n >= 0; --n) {
    const int t0 = n * C, nvalid = min(C, a.T - t0);
    const size_t row0 = (size_t)b * a.T + t0;
    const int kap = nx_meta.x, fmt = nx_meta.y;
    const bool f16 = fmt == FMT_F16;
    Rows<D, true> rows;
    rows.load(a, row0, h, j, nvalid, tid);
    // ---- row scalars; the largest inv of the chunk and the largest entry of the adjoint decide 2^al
    if (tid < C) {
      s_inv[tid] = nx_inv;
      s_dl[tid] = nx_dl * osc;
      const float m = warp_max(fabsf(nx_inv));
      if (lane == 0) atomicMax(const_cast<int*>(&s_fl[3]), __float_as_int(m < 1.0e30f ? m : 1.0e30f));
    }
    if (tid >= C && tid < C + D) s_z[tid - C] = nx_z;
    if (n < nch - 1 && st_thr) {
      const float f = ex2f(fmaxf(s_pe[row], -126.f));
      float m = 0.f, s[32];
#pragma unroll 1
      for (int c0 = cg * SW; c0 < (cg + 1) * SW; c0 += 32) {
        tmem_ld32(lane_base + F::R_R + c0, s);
        tmem_wait_ld();
#pragma unroll
        for (int i = 0; i < 32; ++i) m = fmaxf(m, fabsf(s[i]));
      }
      m = warp_max(m * f);
      if (lane == 0) atomicMax(const_cast<int*>(&s_fl[4]), __float_as_int(m < 1.0e30f ? m : 1.0e30f));
    }
    gate_pass<D>(a, gates, nvalid, s_x, s_bm, s_ft, const_cast<int*>(&s_fl[2]), tid);  // (two barriers)
    int al = min(5 - exp_above(fmaxf(__int_as_float(s_fl[3]), 1e-30f)), 10 - kap);
    const float rm = __int_as_float(s_fl[4]);
    if (rm > 0.f) al = min(al, al_prev + 14 - exp_above(rm));
    al = max(al, -100);
    const float asc = pow2i(al), ksc = pow2i(kap);
    // ---- operands: qn, ks (two-term), v, dO; partial sums of r
    float rp[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) rp[i] = 0.f;
#pragma unroll
    for (int it = 0; it < 2; ++it) {
      const int idx = tid + it * F::THREADS, o = idx % F::OCT, r = idx / F::OCT;  // (o is the same both times)
      float q[8], k[8], vv[8], g[8], x[8];
      rows.f8(rows.q[it], q);
      rows.f8(rows.k[it], k);
      unpack8b(rows.v[it], vv);
      unpack8b(rows.g[it], g);
      load_row8(s_x + r * D + o * 8, x);
      const float inv = s_inv[r] * asc, dl = s_dl[r];
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        q[i] *= ex2f(x[i]) * inv;
        k[i] *= ex2f(-x[i]) * ksc;
        g[i] *= osc;
        rp[i] = fmaf(-dl, q[i], rp[i]);
      }
      uint4 hi, lo;
      const uint32_t at = toff(F::SL_T, r, o * 8);
      split8h(q, f16, hi, lo);
      *reinterpret_cast<uint4*>(sg + F::R_QS + at) = hi;
      *reinterpret_cast<uint4*>(sg + F::R_QS + F::T_TOK + at) = lo;
      split8h(k, f16, hi, lo);
      *reinterpret_cast<uint4*>(sg + F::R_KS + at) = hi;
      *reinterpret_cast<uint4*>(sg + F::R_KS + F::T_TOK + at) = lo;
      *reinterpret_cast<uint4*>(sg + F::R_V + at) = pack8h(vv, f16);
      *reinterpret_cast<uint4*>(sg + F::R_DO + at) = pack8h(g, f16);
    }
#pragma unroll
    for (int off = F::OCT; off < 32; off <<= 1) {  // (the lanes of a warp that hold the same channels)
#pragma unroll
      for (int i = 0; i < 8; ++i) rp[i] += __shfl_xor_sync(0xffffffffu, rp[i], off);
    }
    if (lane < F::OCT) store_row8(s_rp + warp * D + lane * 8, rp);
    publish();
    if (tid == 0) {
      // the state operand of this chunk (needed behind the mask pass), over the exponents
      if (!s_fl[1]) {
        mbar_arrive_expect_tx(bar_s, 2 * F::T_C);
        const uint8_t* src = a.s16 + ((size_t)bh * nch + n) * (2 * F::T_C);
        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(sb + F::R_S),
                     "l"(src), "r"(2 * F::T_C), "r"(bar_s)
                     : "memory");
        copied = nch - 1 - n;
      }
    }
    if (warp == 0 && elect_one()) {
      mm.split(F::R_P, KV(F::R_QS, F::SL_T), KV(F::R_QS + F::T_TOK, F::SL_T), 2 * F::SL_T, KV(F::R_KS, F::SL_T),
               KV(F::R_KS + F::T_TOK, F::SL_T), 2 * F::SL_T, D / 16, instr_desc(128, C, fmt, MAJOR_K, MAJOR_K), false);
      mm.chain(F::R_EP, KV(F::R_DO, F::SL_T), 2 * F::SL_T, KV(F::R_V, F::SL_T), 2 * F::SL_T, D / 16,
               instr_desc(128, C, fmt, MAJOR_K, MAJOR_K), false);
      mma_commit(bar);
    }
    // factor that brings the adjoint behind the chunk to 2^ft R 2^(al + sc)
    const float rfac = pow2i(al - al_prev);
    if (tid < D) {
      const float w = ex2f(fmaxf(s_pe[tid] + s_ft[tid], -126.f)) * rfac * s_r[tid];
      float p = 0.f;
#pragma unroll
      for (int i = 0; i < NW; ++i) p += s_rp[i * D + tid];
      s_r16[tid] = w;
      s_r[tid] = w + p;
    }
    wt.wait();
    if (tid == 0) s_fl[2] = s_fl[3] = s_fl[4] = 0;  // (read by everybody before the barrier in front of the products)
    // ---- mask: P' and E = dO v^T - delta, two-term
    if (tok_thr) {
      const float dl = s_dl[row];
      float s[16], e[16];
      uint4 hi, lo;
#pragma unroll 1
      for (int c0 = cg * TW; c0 < (cg + 1) * TW; c0 += 16) {
        tmem_ld16(lane_base + F::R_P + c0, s);
        tmem_ld16(lane_base + F::R_EP + c0, e);
        tmem_wait_ld();
#pragma unroll
        for (int i8 = 0; i8 < 16; i8 += 8) {
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const bool on = c0 + i8 + i <= row;
            s[i8 + i] = on ? s[i8 + i] : 0.f;
            e[i8 + i] = on ? e[i8 + i] - dl : 0.f;
          }
          const uint32_t at = toff(F::SL_U, row, c0 + i8);
          split8h(s + i8, f16, hi, lo);
          *reinterpret_cast<uint4*>(sg + F::R_PM + at) = hi;
          *reinterpret_cast<uint4*>(sg + F::R_PM + F::T_P + at) = lo;
          split8h(e + i8, f16, hi, lo);
          *reinterpret_cast<uint4*>(sg + F::R_E + at) = hi;
          *reinterpret_cast<uint4*>(sg + F::R_E + F::T_P + at) = lo;
        }
      }
    }
    publish();
    const uint32_t ID_KM = instr_desc(128, D, fmt, MAJOR_K, MAJOR_MN), ID_MM = instr_desc(128, D, fmt, MAJOR_MN, MAJOR_MN),
                   ID_KK = instr_desc(128, D, fmt, MAJOR_K, MAJOR_K);
    if (warp == 0) ws.wait();  // the state operand has landed
    if (warp == 0 && elect_one()) {
      mm.split(F::R_DQ, KV(F::R_E, F::SL_U), KV(F::R_E + F::T_P, F::SL_U), 2 * F::SL_U, MV(F::R_KS, F::SL_T),
               MV(F::R_KS + F::T_TOK, F::SL_T), 256, C / 16, ID_KM, false);
      mm.split(F::R_DQ, KV(F::R_DO, F::SL_T), 0, 2 * F::SL_T, KV(F::R_S, F::SL_C), KV(F::R_S + F::T_C, F::SL_C), 2 * F::SL_C,
               D / 16, ID_KK, true);
      mm.split(F::R_DK, MV(F::R_E, F::SL_U), MV(F::R_E + F::T_P, F::SL_U), 256, MV(F::R_QS, F::SL_T),
               MV(F::R_QS + F::T_TOK, F::SL_T), 256, C / 16, ID_MM, false);
      mm.split(F::R_DVC, MV(F::R_PM, F::SL_U), MV(F::R_PM + F::T_P, F::SL_U), 256, MV(F::R_DO, F::SL_T), 0, 256, C / 16, ID_MM,
               false);
      mma_commit(bar);
    }
    if (tid == 32 && n > 0) prefetch_chunk(maps, b, h, j, t0 - C);
    wt.wait();
    // ---- adjoint pass, over the consumed state operand
    if (st_thr) {
      const float f = ex2f(fmaxf(s_pe[row] + s_ft[row], -126.f)) * rfac;
      float y[32];
      uint4 hi, lo;
      tmem_ld32(lane_base + F::R_R + cg * SW, y);
      tmem_wait_ld();
#pragma unroll
      for (int i8 = 0; i8 < 32; i8 += 8) {
#pragma unroll
        for (int i = 0; i < 8; ++i) y[i8 + i] *= f;
        split8h(y + i8, f16, hi, lo);
        *reinterpret_cast<uint4*>(sg + F::R_S + toff(F::SL_C, row, cg * SW + i8)) = hi;
        *reinterpret_cast<uint4*>(sg + F::R_S + F::T_C + toff(F::SL_C, row, cg * SW + i8)) = lo;
      }
      tmem_st32(lane_base + F::R_R + cg * SW, y);
      tmem_wait_st();
    }
    publish();
    if (warp == 0 && elect_one()) {
      mm.split(F::R_DK, KV(F::R_V, F::SL_T), 0, 2 * F::SL_T, KV(F::R_S, F::SL_C), KV(F::R_S + F::T_C, F::SL_C), 2 * F::SL_C,
               D / 16, ID_KK, true);
      mm.split(F::R_DVC, KV(F::R_KS, F::SL_T), KV(F::R_KS + F::T_TOK, F::SL_T), 2 * F::SL_T, MV(F::R_S, F::SL_C),
               MV(F::R_S + F::T_C, F::SL_C), 256, D / 16, ID_KM, true);
      mm.split(F::R_R, MV(F::R_QS, F::SL_T), MV(F::R_QS + F::T_TOK, F::SL_T), 256, MV(F::R_DO, F::SL_T), 0, 256, C / 16, ID_MM,
               true);
      mma_commit(bar);
    }
    fetch_next(n - 1);
    for (int i = tid; i < D; i += F::THREADS) s_pe[i] = s_bm[i];  // (read again behind the next barrier at the earliest)
    wt.wait();
    // ---- wq, wk, dv of the chunk's rows into fp32 tiles over the dead operands
    const float usc = pow2i(-(al + kap + sc));
    static_assert(SW == 32, "32 columns per thread");
    if (tok_thr) {
      const float dl = s_dl[row];
#pragma unroll
      for (int i16 = 0; i16 < SW; i16 += 16) {
        float dq[16], dk[16];
        tmem_ld16(lane_base + F::R_DQ + cg * SW + i16, dq);
        tmem_ld16(lane_base + F::R_DK + cg * SW + i16, dk);
        tmem_wait_ld();
#pragma unroll
        for (int i8 = 0; i8 < 16; i8 += 8) {
          const int c0 = cg * SW + i16 + i8;
          float hi[8], lo[8];
          const uint32_t at = toff(F::SL_T, row, c0);
          unpack8h(*reinterpret_cast<const uint4*>(sg + F::R_QS + at), f16, hi);
          unpack8h(*reinterpret_cast<const uint4*>(sg + F::R_QS + F::T_TOK + at), f16, lo);
#pragma unroll
          for (int i = 0; i < 8; ++i) dq[i8 + i] = (hi[i] + lo[i]) * fmaf(-dl, s_z[c0 + i], dq[i8 + i]) * usc;
          unpack8h(*reinterpret_cast<const uint4*>(sg + F::R_KS + at), f16, hi);
          unpack8h(*reinterpret_cast<const uint4*>(sg + F::R_KS + F::T_TOK + at), f16, lo);
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            dk[i8 + i] = (hi[i] + lo[i]) * (dk[i8 + i] + s_r16[c0 + i]) * usc;
            wmax = fmaxf(wmax, fmaxf(fabsf(dq[i8 + i]), fabsf(dk[i8 + i])));
          }
#pragma unroll
          for (int i = 0; i < 8; i += 4) {
            *reinterpret_cast<float4*>(sg + F::R_WQ + foff(row, (c0 + i) >> 2)) = make_float4(dq[i8 + i], dq[i8 + i + 1], dq[i8 + i + 2], dq[i8 + i + 3]);
            *reinterpret_cast<float4*>(sg + F::R_WK + foff(row, (c0 + i) >> 2)) = make_float4(dk[i8 + i], dk[i8 + i + 1], dk[i8 + i + 2], dk[i8 + i + 3]);
          }
        }
      }
      {
        float d[32];
        tmem_ld32(lane_base + F::R_DVC + cg * SW, d);
        tmem_wait_ld();
#pragma unroll
        for (int i = 0; i < 32; i += 4)
          *reinterpret_cast<float4*>(sg + F::R_DV + foff(row, (cg * SW + i) >> 2)) = make_float4(d[i] * usc, d[i + 1] * usc, d[i + 2] * usc, d[i + 3] * usc);
      }
    }
    publish();
    if (tid == 0) {  // whole rows to memory by the copy engine (rows past the end are clipped)
#pragma unroll 1
      for (int c0 = 0; c0 < D; c0 += 32) {
        tma_store_4d(&maps.wq, sb + F::R_WQ + c0 * (C * 4), c0, h, t0, b);
        tma_store_4d(&maps.wk, sb + F::R_WK + c0 * (C * 4), c0, h, t0, b);
        tma_store_4d(&maps.dvh, sb + F::R_DV + c0 * (C * 4), c0, h, t0, b);
      }
      tma_store_commit();
    }
    uint4 graw[2];  // this chunk's gate again, for the derivative of the log-decays
#pragma unroll
    for (int it = 0; it < 2; ++it) {
      const int idx = tid + it * F::THREADS, o = idx % F::OCT, r = idx / F::OCT;
      if (a.gate_dim != 1 && r < nvalid) graw[it] = *reinterpret_cast<const uint4*>(a.gate + ((row0 + r) * a.H + h) * D + o * 8);
    }
    // ---- gate gradient: reverse running sum of wq - wk over the chunk's tokens on top of what lies behind it; thread =
    // (channel, run of tokens); the runs' totals meet in shared memory
    {
      constexpr int RUNS = F::THREADS / D, RT = C / RUNS;  // 4 runs of 16 tokens
      const int c = tid % D, run = tid / D;
      float v[RT], acc = 0.f;
#pragma unroll
      for (int i = RT - 1; i >= 0; --i) {
        const uint32_t at = foff(run * RT + i, c >> 2) + (c & 3) * 4;
        acc += *reinterpret_cast<const float*>(sg + F::R_WQ + at) - *reinterpret_cast<const float*>(sg + F::R_WK + at);
        v[i] = acc;
      }
      s_rp[run * D + c] = acc;  // (NW >= RUNS rows)
      __syncthreads();
      float off = s_car[c], all = off;
#pragma unroll
      for (int r = RUNS - 1; r >= 0; --r) {
        const float t = s_rp[r * D + c];
        if (r > run) off += t;
        all += t;
      }
#pragma unroll
      for (int i = 0; i < RT; ++i) *reinterpret_cast<float*>(sg + F::R_DG + foff(run * RT + i, c >> 2) + (c & 3) * 4) = v[i] + off;
      __syncthreads();
      if (run == 0) s_car[c] = all;
    }
    // d(log-decay) / d(gate entry): 1 - sigmoid(a) = 1 / (1 + e^a)
    auto dlog = [&](float av) {
      return a.gate_mode == LAWCAT_GATE_LOGDECAY ? 1.f : rcpf(1.f + ex2f(fminf(av * 1.4426950408889634f, 126.f))) * a.inv_tau;
    };
    if (a.gate_dim == 1) {
      for (int r = warp; r < nvalid; r += NW) {
        float s = 0.f;
        for (int c = lane; c < D; c += 32) s += *reinterpret_cast<const float*>(sg + F::R_DG + foff(r, c >> 2) + (c & 3) * 4);
        s = warp_sum(s);
        if (lane == 0) {
          const size_t gi = (row0 + r) * a.H + h;
          a.dgate[gi] = __float2bfloat16_rn(s * dlog(__bfloat162float(a.gate[gi])));
        }
      }
    } else {
#pragma unroll
      for (int it = 0; it < 2; ++it) {
        const int idx = tid + it * F::THREADS, o = idx % F::OCT, r = idx / F::OCT;
        if (r >= nvalid) continue;
        float av[8], d[8];
        unpack8b(graw[it], av);
        const float4 x = *reinterpret_cast<const float4*>(sg + F::R_DG + foff(r, 2 * o)), y = *reinterpret_cast<const float4*>(sg + F::R_DG + foff(r, 2 * o + 1));
        d[0] = x.x; d[1] = x.y; d[2] = x.z; d[3] = x.w; d[4] = y.x; d[5] = y.y; d[6] = y.z; d[7] = y.w;
#pragma unroll
        for (int i = 0; i < 8; ++i) d[i] *= dlog(av[i]);
        store_row8(a.dgate + ((row0 + r) * a.H + h) * D + o * 8, d);
      }
    }
    al_prev = al;
    if (tid == 0) tma_store_wait_read();  // (the next chunk writes over the result tiles)
    __syncthreads();
  }
  wmax = warp_max(wmax);
  if (lane == 0) atomicMax(const_cast<int*>(&s_fl[5]), __float_as_int(wmax < 1.0e30f ? wmax : 1.0e30f));
  tc_fence_before_sync();
  __syncthreads();
  if (tid == 0) {
    a.wmax[bh] = __int_as_float(s_fl[5]);
    tma_store_wait_all();
    if (s_fl[1] && copied >= 0) mbar_wait(bar_s, (uint32_t)(copied & 1));  // (after a wait that ran out it may still be under way)
  }
  if (warp == 0) {
    tc_fence_after_sync();
    tmem_dealloc(mm.tmem, F::COLS);
  }
}

// ------------------------------------------------------------------------------------------------ mix backward
// From w = p * dp of both streams (p the features) back through the softmax and the shared linear layer:
//   dy = w - p sum(w),   du = dy W_h^T (query stream; key stream summed over the heads of the group),   dW_h += u^T dy
// One block = one (batch, key head, tile of 128 tokens), walking the group's heads and both streams. dy (scaled by a power of
// two from the largest |w| of the group, or of the head where that is far smaller) and u, the recomputed conv output, are
// two-term fp16 pairs; the key stream's du is accumulated over the heads in tensor memory. du of the query stream overwrites wq
// in place.
// What bounds it is the chain loads -> operands -> products -> gradients out of a step (head, stream). It is folded: while a step's
// products run, the block works out the next step's operands in registers (its loads are what waits, not the tensor cores), and the
// gradients of the step before leave tensor memory (dW has two accumulators, du of the query stream is not needed before the next
// head's products).
struct MArgs {
  const bf16 *q, *k, *w_q, *w_k, *W, *cache_q, *cache_k;
  const float *qd, *kd, *wk;
  float *wq;                 // in: wq; out: du of the query stream
  float *du_k, *dW;          // [B,T,Hkv,D]; [H,D,D] (atomic adds into zeros)
  const float* wmax;
  int* dev_status;
  int B, T, H, Hkv, K;
  int parts;                 // blocks that share a group's heads; more than one: du_k is added to (zeroed by the sweep)
};

template <int D>
struct MCfg {
  using L = Lay<D>;
  static constexpr int THREADS = D == 128 ? 512 : 256, NCG = THREADS / 128;  // (16 warps per SM either way)
  static constexpr uint32_t WT = 0, U = L::TILE_W, DY = U + 2 * L::TILE_U, ST = DY + 2 * L::TILE_U;  // ST: 64 columns of fp32 rows on their way out
  static constexpr uint32_t ST_ROW = 272, TAPS = ST + TT * ST_ROW, BAR = TAPS + 2 * D * 16;                              // taps of two steps
  static constexpr uint32_t BYTES = BAR + 64;
  static constexpr uint32_t DUQ = 0, DUK = D, DWC = 2 * D, COLS = 4 * D;  // (DWC: two accumulators)
};

template <int D>
__global__ void __launch_bounds__(MCfg<D>::THREADS, D == 128 ? 1 : 2) mix_bwd_kernel(const MArgs a) {
  using L = Lay<D>;
  using M = MCfg<D>;
  extern __shared__ __align__(128) uint8_t sg[];
  const uint32_t sb = smem_u32(sg);
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  volatile int* const s_fl = reinterpret_cast<volatile int*>(sg + M::BAR + 16);  // tmem base, abort
  const int part = blockIdx.x % a.parts, t0 = blockIdx.x / a.parts * TT, bj = blockIdx.z * gridDim.y + blockIdx.y, j = bj % a.Hkv, b = bj / a.Hkv, G = a.H / a.Hkv;
  if (b >= a.B) return;
  const int nvalid = min(TT, a.T - t0);
  if (tid == 0) {
    mbar_init(sb + M::BAR, 1);
    mbar_fence_init();
    s_fl[1] = 0;
  }
  if (warp == 0) {
    tmem_alloc(sb + M::BAR + 16, M::COLS);
    tmem_relinquish();
  }
  asm volatile("griddepcontrol.wait;" ::: "memory");
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const Mma mm{(uint32_t)s_fl[0]};
  const uint32_t lane_base = mm.tmem + ((uint32_t)((warp & 3) * 32) << 16);
  const int row = (warp & 3) * 32 + lane, cg = warp >> 2;
  constexpr int HC = D / M::NCG, NTH = M::THREADS;
  Waiter wt{sb + M::BAR, 0u, s_fl + 1, a.dev_status};
  // 2^sg on dy. The group's largest |w| becomes 2^7 .. 2^8 by it, which leaves |dy| <= |w| + sum |w| below the fp16 maximum for
  // every row. A head more than 2^4 below the others gets a power of two of its own (`spread`: there is one).
  auto sg_of = [](float w) -> int { return 8 - exp_above(fmaxf(w, 1e-30f)); };
  const float* const wmax = a.wmax + b * a.H + j * G;
  float whi = 0.f, wlo = -1e30f;  // (wlo: minus the smallest)
  for (int g = lane; g < G; g += 32) {
    const float w = wmax[g];
    whi = fmaxf(whi, w);
    wlo = fmaxf(wlo, -w);
  }
  const int sg_group = sg_of(warp_max(whi));
  const bool spread = __any_sync(0xffffffffu, sg_of(-warp_max(wlo)) - sg_group > 4);
  auto scale_of = [&](int g) -> int {
    if (!spread) return sg_group;
    const int own = sg_of(wmax[g]);
    return own - sg_group <= 4 ? sg_group : min(own, sg_group + 60);
  };
  const int o = tid % L::OPR, rr0 = tid / L::OPR;
  constexpr int RSTEP = NTH / L::OPR, RPT = TT / RSTEP, WPT = D * L::OPR / NTH;
  // fp32 accumulators leave 64 columns at a time through the staging tile (rows of 272 bytes: the lanes that write own rows)
  auto stage = [&](uint32_t col, int h64, float isc) {
    if (cg * HC >= h64 && cg * HC < h64 + 64) {  // (whole warps)
      float d[16];
#pragma unroll 1
      for (int c0 = cg * HC; c0 < (cg + 1) * HC; c0 += 16) {
        tmem_ld16(lane_base + col + c0, d);
        tmem_wait_ld();
#pragma unroll
        for (int i = 0; i < 16; i += 4)
          *reinterpret_cast<float4*>(sg + M::ST + row * M::ST_ROW + (c0 - h64 + i) * 4) = make_float4(d[i] * isc, d[i + 1] * isc, d[i + 2] * isc, d[i + 3] * isc);
      }
    }
  };
  // du. Width 64: the bulk-copy engine takes the rows on from the staging tile, behind the block's other work (8 x 1024 tokens: the
  // kernel 131 us; 138 by the threads). Width 128, where a tile is two trips through staging that would wait for one another: by the
  // threads (4 x 1300 tokens: 238 us; 244).
  auto du_out = [&](uint32_t col, float* dst, int NH, int head, float isc, bool add) {
    if constexpr (D == 64) {
      stage(col, 0, isc);
      fence_proxy_async();
      __syncthreads();
      if (tid < nvalid) {
        float* const p = dst + (((size_t)b * a.T + t0 + tid) * NH + head) * D;
        if (add) asm volatile("cp.reduce.async.bulk.global.shared::cta.bulk_group.add.f32 [%0], [%1], 256;" ::"l"(p), "r"(sb + M::ST + tid * M::ST_ROW) : "memory");
        else asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], 256;" ::"l"(p), "r"(sb + M::ST + tid * M::ST_ROW) : "memory");
        tma_store_commit();
      }
    } else {
#pragma unroll 1
      for (int h64 = 0; h64 < D; h64 += 64) {
        stage(col, h64, isc);
        __syncthreads();
#pragma unroll 4
        for (int idx = tid; idx < nvalid * 16; idx += NTH) {
          const int pc = idx % 16, r = idx / 16;
          float* const p = dst + (((size_t)b * a.T + t0 + r) * NH + head) * D + h64 + pc * 4;
          const float4 v = *reinterpret_cast<const float4*>(sg + M::ST + r * M::ST_ROW + pc * 16);
          if (add) asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
          else *reinterpret_cast<float4*>(p) = v;
        }
        __syncthreads();
      }
    }
  };
  // dW of a head, row c of the accumulator being row c of dW. Width 64: the bulk-copy engine adds the rows, behind the block's other
  // work. Width 128, where a row would be two trips through the staging tile: added from where they are.
  auto dw_out = [&](int g) {
    if (!a.dW) return;
    float* const dst = a.dW + ((size_t)(j * G + g) * D + (row < D ? row : 0)) * D;
    const float isc = pow2i(-scale_of(g));
    if constexpr (D == 64) {
      stage(M::DWC + (g & 1) * D, 0, isc);
      fence_proxy_async();
      __syncthreads();
      if (tid < D) {
        asm volatile("cp.reduce.async.bulk.global.shared::cta.bulk_group.add.f32 [%0], [%1], 256;" ::"l"(dst), "r"(sb + M::ST + tid * M::ST_ROW) : "memory");
        tma_store_commit();
      }
    } else {
      float d[8];
#pragma unroll 1
      for (int c0 = cg * HC; c0 < (cg + 1) * HC; c0 += 8) {
        tmem_ld8(lane_base + M::DWC + (g & 1) * D + c0, d);
        tmem_wait_ld();
#pragma unroll
        for (int i = 0; i < 8; i += 4)
          asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(dst + c0 + i), "f"(d[i] * isc), "f"(d[i + 1] * isc),
                       "f"(d[i + 2] * isc), "f"(d[i + 3] * isc)
                       : "memory");
      }
    }
  };
  // this block's steps: those of heads [G part / parts, G (part + 1) / parts) of the group
  const int s_begin = 2 * (G * part / a.parts), s_end = 2 * (G * (part + 1) / a.parts);
  auto taps = [&](int s) {  // of step s into its slot
    if (s < s_end) load_taps<D>(sg + M::TAPS + (s & 1) * D * 16, s & 1 ? a.w_k : a.w_q, s & 1 ? j : j * G + (s >> 1), a.K, tid, NTH);
  };
  uint4 dyh[RPT], dyl[RPT], uh[RPT], ul[RPT];  // a step's operands: this thread's octets of dy and u, hi and lo
  auto operands = [&](int s) {
    const int g = s >> 1, stream = s & 1, h = j * G + g;
    const float sc = pow2i(scale_of(g));
    const float* wp = stream ? a.wk : a.wq;
    const float* pp = stream ? a.kd : a.qd;
    float4 wr[RPT][2], pr[RPT][2];  // (all loads of a step in flight together: they are what a step takes longest over)
#pragma unroll
    for (int k = 0; k < RPT; ++k) {
      const int r = rr0 + k * RSTEP;
      const size_t at = (((size_t)b * a.T + t0 + min(r, nvalid - 1)) * a.H + h) * D + o * 8;
      load_octet(wp + at, wr[k]);
      load_octet(pp + at, pr[k]);
    }
    uint4 raw[RPT + HALO];
    conv_load<D, RPT>(raw, stream ? a.k : a.q, stream ? a.cache_k : a.cache_q, b, t0 + rr0 * RPT, a.T, stream ? a.Hkv : a.H, stream ? j : h, a.K, o);
    // the rows of the step behind travel towards L2 meanwhile
    if (s + 1 < s_end) {
      const int nh = h + stream;
      const float* wn = stream ? a.wq : a.wk;
      const float* pn = stream ? a.qd : a.kd;
      constexpr int LF = D * 4 / 128;
      for (int idx = tid; idx < nvalid * 2 * LF; idx += NTH) {
        const int r = idx / (2 * LF), l = idx % (2 * LF);
        prefetch_l2((l < LF ? wn : pn) + (((size_t)b * a.T + t0 + r) * a.H + nh) * D + (l % LF) * 32);
      }
      if (stream && tid < nvalid) {
        const bf16* xn = a.q + (((size_t)b * a.T + t0 + tid) * a.H + nh) * D;
        prefetch_l2(xn);
        if (D == 128) prefetch_l2(xn + 64);
      }
    }
#pragma unroll
    for (int k = 0; k < RPT; ++k) {
      const float on = rr0 + k * RSTEP < nvalid ? sc : 0.f;
      float wv[8] = {wr[k][0].x, wr[k][0].y, wr[k][0].z, wr[k][0].w, wr[k][1].x, wr[k][1].y, wr[k][1].z, wr[k][1].w};
      const float pv[8] = {pr[k][0].x, pr[k][0].y, pr[k][0].z, pr[k][0].w, pr[k][1].x, pr[k][1].y, pr[k][1].z, pr[k][1].w};
      float s8 = 0.f;
#pragma unroll
      for (int i = 0; i < 8; ++i) s8 += wv[i];
#pragma unroll
      for (int off = 1; off < L::OPR; off <<= 1) s8 += __shfl_xor_sync(0xffffffffu, s8, off);
#pragma unroll
      for (int i = 0; i < 8; ++i) wv[i] = on != 0.f ? fmaf(-pv[i], s8, wv[i]) * on : 0.f;
      split8h(wv, true, dyh[k], dyl[k]);
    }
    conv_emit<D, RPT>(raw, sg + M::TAPS + stream * D * 16, o, [&](int i, const uint64_t* u2) {
      float u[8];
      pairs_to_floats(u2, u);
      split8h(u, true, uh[i], ul[i]);
    });
  };
  taps(s_begin);
  load_w_tile<D>(sg + M::WT, a.W + ((size_t)j * G + (s_begin >> 1)) * D * D, tid, NTH);
  __syncthreads();
  operands(s_begin);
  int sg_at = scale_of(s_begin >> 1);  // power of two on the key stream's du so far
#pragma unroll 1
  for (int s = s_begin; s < s_end; ++s) {
    const int g = s >> 1, stream = s & 1, h = j * G + g;
    uint4 wreg[WPT];
    const bool next_w = stream == 0 && s > s_begin;
    if (next_w) {
#pragma unroll
      for (int k = 0; k < WPT; ++k) wreg[k] = *reinterpret_cast<const uint4*>(a.W + (size_t)h * D * D + (size_t)(tid + k * NTH) * 8);
    }
    if (s > s_begin) wt.wait();  // the products of the step in front: its operands and W_h have been read
    if (next_w) {
#pragma unroll
      for (int k = 0; k < WPT; ++k) {
        const int idx = tid + k * NTH;
        float f[8];
        unpack8b(wreg[k], f);
        *reinterpret_cast<uint4*>(sg + M::WT + toff(L::SLAB_W, idx / L::OPR, idx % L::OPR * 8)) = pack8f16(f);
      }
    }
#pragma unroll
    for (int k = 0; k < RPT; ++k) {
      const uint32_t ady = toff(L::SLAB_U, rr0 + k * RSTEP, o * 8), au = toff(L::SLAB_U, rr0 * RPT + k, o * 8);
      *reinterpret_cast<uint4*>(sg + M::DY + ady) = dyh[k];
      *reinterpret_cast<uint4*>(sg + M::DY + L::TILE_U + ady) = dyl[k];
      *reinterpret_cast<uint4*>(sg + M::U + au) = uh[k];
      *reinterpret_cast<uint4*>(sg + M::U + L::TILE_U + au) = ul[k];
    }
    const int sgm = scale_of(g);
    if (stream == 0 && sgm != sg_at) {  // the key stream's du so far, on this head's scale (the choice of powers is uniform)
      if (s > s_begin) {
        const float f = pow2i(sgm - sg_at);
        float d[8];
#pragma unroll 1
        for (int c0 = cg * HC; c0 < (cg + 1) * HC; c0 += 8) {
          tmem_ld8(lane_base + M::DUK + c0, d);
          tmem_wait_ld();
#pragma unroll
          for (int i = 0; i < 8; ++i) d[i] *= f;
          tmem_st8(lane_base + M::DUK + c0, d);
        }
        tmem_wait_st();
      }
      sg_at = sgm;
    }
    taps(s + 1);
    if (D == 64 && tid < TT) tma_store_wait_read();  // (the rows of the step in front have left the staging tile)
    fence_proxy_async();
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
    if (warp == 0 && elect_one()) {
      mm.split(stream ? M::DUK : M::DUQ, kview(sb + M::DY, L::SLAB_U), kview(sb + M::DY + L::TILE_U, L::SLAB_U), 2 * L::SLAB_U,
               kview(sb + M::WT, L::SLAB_W), 0, 2 * L::SLAB_W, D / 16, instr_desc(128, D, FMT_F16, MAJOR_K, MAJOR_K),
               stream == 1 && s > s_begin + 1);
      mm.split(M::DWC + (g & 1) * D, mview(sb + M::U, L::SLAB_U), mview(sb + M::U + L::TILE_U, L::SLAB_U), 256, mview(sb + M::DY, L::SLAB_U),
               mview(sb + M::DY + L::TILE_U, L::SLAB_U), 256, TT / 16, instr_desc(128, D, FMT_F16, MAJOR_MN, MAJOR_MN), stream == 1);
      mma_commit(sb + M::BAR);
    }
    if (stream) du_out(M::DUQ, a.wq, a.H, h, pow2i(-sgm), false);
    else if (s > s_begin) dw_out(g - 1);
    if (s + 1 < s_end) operands(s + 1);
  }
  wt.wait();
  auto staging_free = [&]() {
    if (D == 64) {
      if (tid < TT) tma_store_wait_read();
      __syncthreads();
    }
  };
  staging_free();
  dw_out((s_end >> 1) - 1);
  staging_free();
  du_out(M::DUK, a.du_k, a.Hkv, j, pow2i(-sg_at), a.parts > 1);
  if (D == 64 && tid < TT) tma_store_wait_all();
  tc_fence_before_sync();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after_sync();
    tmem_dealloc(mm.tmem, M::COLS);
  }
}

// dv[b,t,j,:] = sum over the query heads of group j of the per-head gradients; one thread per 8 channels
// (and zeroes the tap gradients, n0 and n1 floats, for the conv backward that follows)
__global__ void dv_sum_kernel(const float* __restrict__ dvh, bf16* __restrict__ dv, size_t total, int G, int oct, float* z0, int n0,
                              float* z1, int n1) {
  const size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  asm volatile("griddepcontrol.wait;" ::: "memory");
  for (size_t i = idx; i < (size_t)n0 + n1; i += (size_t)gridDim.x * blockDim.x) (i < (size_t)n0 ? z0[i] : z1[i - n0]) = 0.f;
  if (idx >= total) return;
  const size_t btj = idx / oct;
  const int o8 = (int)(idx % oct);
  float s[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  for (int g = 0; g < G; ++g) {
    float x[8];
    load_row8(dvh + ((btj * G + g) * oct + o8) * 8, x);
#pragma unroll
    for (int i = 0; i < 8; ++i) s[i] += x[i];
  }
  store_row8(dv + (btj * oct + o8) * 8, s);
}

struct Plan {
  size_t qd, kd, wq, wk, dvh, du_k, inv, delta, domax, z16, meta, s16, wmax, total;
};
static Plan plan(const lawcat_params& p) {
  Plan L;
  size_t off = 0;
  auto take = [&](size_t n) { const size_t o = off; off += align_up(n, 256); return o; };
  const size_t bth = (size_t)p.B * p.T * p.H, nf = 4 * bth * p.d_k, ch = (size_t)p.B * p.H * ((p.T + C - 1) / C);
  L.qd = take(nf); L.kd = take(nf); L.wq = take(nf); L.wk = take(nf); L.dvh = take(nf);
  L.du_k = take(nf / (p.H / p.H_kv));
  L.inv = take(4 * bth); L.delta = take(4 * bth); L.domax = take(8 * (size_t)p.B * p.H);
  L.z16 = take(4 * ch * p.d_k); L.meta = take(8 * ch); L.s16 = take(ch * 4 * p.d_k * p.d_k); L.wmax = take(4 * (size_t)p.B * p.H);
  L.total = off + 256;  // (the base is rounded up: rows are read 32 bytes at a time)
  return L;
}

// How many blocks of the mix backward share the heads of a group: two where that fills the last round of blocks better (one per SM at
// width 128, two at 64; a block's first operands and last gradients, which nothing hides, are worth about half a head). 4 x 1300 tokens,
// 32/8 heads of 128 (352 blocks, 2.4 rounds): 236 us as one, 219 as two; 8 x 1024 of 64 (512 blocks, 1.7 rounds) stays one.
static int mix_parts(const lawcat_params& p) {
  const int G = p.H / p.H_kv, slots = sm_count() * (p.d_k == 128 ? 1 : 2);
  const long long blocks = (long long)p.B * p.H_kv * ((p.T + TT - 1) / TT);
  int best = 1;
  long long cost = 0;
  for (int n = 1; n <= 2 && n <= G; ++n) {
    const long long c = (blocks * n + slots - 1) / slots * (2 * ((G + n - 1) / n) + 1);
    if (n == 1 || c < cost) { cost = c; best = n; }
  }
  return best;
}

static int raise_limits() {
  static std::mutex mu;
  static bool done[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return LAWCAT_ERR_CUDA;
  std::lock_guard<std::mutex> lk(mu);
  if (done[dev]) return LAWCAT_OK;
  auto up = [](auto* k, uint32_t n) { return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)n) == cudaSuccess; };
  if (!up(sweep_kernel<64>, Cfg<64>::F_BYTES) || !up(sweep_kernel<128>, Cfg<128>::F_BYTES) || !up(reverse_kernel<64>, Cfg<64>::R_BYTES) ||
      !up(reverse_kernel<128>, Cfg<128>::R_BYTES) || !up(mix_bwd_kernel<64>, MCfg<64>::BYTES) || !up(mix_bwd_kernel<128>, MCfg<128>::BYTES))
    return LAWCAT_ERR_CUDA;
  done[dev] = true;
  return LAWCAT_OK;
}

template <int D>
static int run(const Ctx& c, const Args& a, const Maps& maps, const MArgs& m) {
  const lawcat_params& p = *c.p;
  {
    LaunchScope _ls("layer_bwd_sweep", c.stream);
    launch_behind(sweep_kernel<D>, dim3(p.B * p.H), dim3(Cfg<D>::THREADS), Cfg<D>::F_BYTES, c.stream, a, maps);
    LAWCAT_CHECK_LAUNCH();
  }
  {
    LaunchScope _ls("layer_bwd_reverse", c.stream);
    launch_behind(reverse_kernel<D>, dim3(p.B * p.H), dim3(Cfg<D>::THREADS), Cfg<D>::R_BYTES, c.stream, a, maps);
    LAWCAT_CHECK_LAUNCH();
  }
  LaunchScope _ls("layer_bwd_mix", c.stream);
  // (tiles along x, with neighbours on the same head: 3 tiles of 8 heads of 128, head by head 92.7 us instead of 90.6; the y axis
  // ends at 65535, so the heads go on along z)
  const unsigned heads = (unsigned)(p.B * p.H_kv), ny = heads < 32768u ? heads : 32768u;
  launch_behind(mix_bwd_kernel<D>, dim3((unsigned)((p.T + TT - 1) / TT * m.parts), ny, (heads + ny - 1) / ny), dim3(MCfg<D>::THREADS), MCfg<D>::BYTES,
                c.stream, m);
  LAWCAT_CHECK_LAUNCH();
  return LAWCAT_OK;
}

}  // namespace lbt

// (sharp sigmoid gates and short calls: the same exceptions as the forward, see gla_tc_supported)
bool layer_bwd_tc_supported(const lawcat_params& p) {
  const bool sharp = p.gate_mode == LAWCAT_GATE_LOGITS && p.gate_tau < 8.f;
  return p.dtype == LAWCAT_BF16 && (p.d_k == 64 || p.d_k == 128) && p.d_v == p.d_k && (p.gate_dim == p.d_k || p.gate_dim == 1) &&
         !sharp && p.phi == LAWCAT_PHI_SOFTMAX && p.conv_k <= ctc::HALO + 1 && !p.mix_unshared && p.B > 0 && p.T >= 16 &&
         (p.chunk == 0 || p.chunk == lbt::C);
}

size_t layer_bwd_tc_workspace_bytes(const lawcat_params& p) { return lbt::plan(p).total; }

int launch_layer_bwd_tc(const Ctx& c, const void* q, const void* k, const void* v, const void* gate, const void* w_q,
                        const void* w_k, const void* W, const void* cache_q, const void* cache_k, const float* S0,
                        const float* z0, const void* dO, void* dq, void* dk, void* dv, void* dgate, float* dw_q, float* dw_k,
                        float* dW, void* ws) {
  using namespace lbt;
  const lawcat_params& p = *c.p;
  int r = raise_limits();
  if (r) return r;
  const Plan L = plan(p);
  char* w = (char*)align_up((size_t)ws, 256);
  Args a{};
  a.qd = (float*)(w + L.qd); a.kd = (float*)(w + L.kd); a.v = (const bf16*)v; a.gate = (const bf16*)gate; a.dO = (const bf16*)dO;
  a.S0 = S0; a.z0 = z0; a.wq = (float*)(w + L.wq); a.wk = (float*)(w + L.wk); a.dvh = (float*)(w + L.dvh); a.dgate = (bf16*)dgate;
  a.inv = (float*)(w + L.inv); a.delta = (float*)(w + L.delta); a.domax = (float2*)(w + L.domax); a.z16 = (float*)(w + L.z16);
  a.meta = (int*)(w + L.meta); a.s16 = (uint8_t*)(w + L.s16); a.wmax = (float*)(w + L.wmax); a.dW = dW; a.dev_status = c.dev_status;
  a.B = p.B; a.T = p.T; a.H = p.H; a.Hkv = p.H_kv; a.gate_dim = p.gate_dim; a.gate_mode = p.gate_mode; a.normalize = p.normalize;
  a.inv_tau = 1.f / p.gate_tau; a.eps = p.eps;
  MArgs m{(const bf16*)q, (const bf16*)k, (const bf16*)w_q, (const bf16*)w_k, (const bf16*)W, (const bf16*)cache_q,
          (const bf16*)cache_k, a.qd, a.kd, a.wk, a.wq, (float*)(w + L.du_k), dW, a.wmax, c.dev_status, p.B, p.T, p.H, p.H_kv, p.conv_k,
          mix_parts(p)};
  a.du_k = m.parts > 1 ? m.du_k : nullptr;
  if ((r = launch_convmix_tc_fwd(c, q, k, w_q, w_k, W, cache_q, cache_k, (void*)a.qd, (void*)a.kd, true))) return r;
  Maps maps;
  const int D = p.d_k;
  if (!tensor_map(&maps.qd, a.qd, true, p.H, p.T, p.B, D, D, C, false) || !tensor_map(&maps.kd, a.kd, true, p.H, p.T, p.B, D, D, C, false) ||
      !tensor_map(&maps.v, v, false, p.H_kv, p.T, p.B, D, D, C, false) || !tensor_map(&maps.dO, dO, false, p.H, p.T, p.B, D, D, C, false) ||
      !tensor_map(&maps.wq, a.wq, true, p.H, p.T, p.B, D, 32, C, true) || !tensor_map(&maps.wk, a.wk, true, p.H, p.T, p.B, D, 32, C, true) ||
      !tensor_map(&maps.dvh, a.dvh, true, p.H, p.T, p.B, D, 32, C, true))
    return LAWCAT_ERR_CUDA;
  if ((r = D == 64 ? run<64>(c, a, maps, m) : run<128>(c, a, maps, m))) return r;
  {
    const int oct = p.d_v / 8;
    const size_t total = (size_t)p.B * p.T * p.H_kv * oct;
    LaunchScope _ls("dv_sum", c.stream);
    launch_behind(dv_sum_kernel, dim3((unsigned)((total + 255) / 256)), dim3(256), 0, c.stream, (const float*)a.dvh, (bf16*)dv, total,
                  p.H / p.H_kv, oct, dw_q, dw_q ? p.H * p.d_k * p.conv_k : 0, dw_k, dw_k ? p.H_kv * p.d_k * p.conv_k : 0);
    LAWCAT_CHECK_LAUNCH();
  }
  return launch_conv_only_bwd(c, q, k, w_q, w_k, cache_q, cache_k, a.wq, m.du_k, dq, dk, dw_q, dw_k);
}

}  // namespace lawcat
