// The state-only pass of the layer forward: the end state [S | z] and the total decay of a piece of a sequence that starts from
// a zero state (conv, mix and softmax of the key stream, gate, state update; no query stream, no output). The segments of a long
// sequence get their start states from these (layer_tc.cu).
//
// Everything is transposed against the layer kernel: tensor-memory lane = key channel, column = token. The mix is Y^T = W_h^T u^T
// (all 128 rows of the product are channels in use, where the layer kernel's stacked tile would have 64 key rows), a thread owns
// one channel of half a chunk's tokens, and what belongs to a channel stays with it in registers: its log-decays, the exponents
// b_C - b_i (so that kh_i = phi_i 2^(b_C - b_i) needs no other reference token), its features, its row of the state and of z. kh
// goes into tensor memory as the A operand of the state update, S += kh v. No exponent tile, no kh tile, no hand-over between
// warps through shared memory; only the softmax crosses lanes, through a max reduction per token and a folding sum.
// One block is lock-step with two barriers a chunk; 105 KB of shared memory and 256 tensor-memory columns let two blocks share
// an SM, and one fills the other's waits: 4.4k cycles a chunk and SM (6.8k as a mode of the layer kernel, one block per SM).
// Bound by instruction issue (10.2k warp instructions a chunk, 46 % of the slots) and shared-memory latency; the
// special-function unit, four operations an entry, is at 38 %. 32 heads of 128, 32768 tokens: 323 -> 232 us; 32 heads of 64, 8192
// tokens: 62.8 -> 47.7; 32 heads of 128, 1223 tokens: 31.4 -> 24.3. (With the row's maximum in front of the exponentials and four
// barriers: 247, 49.2, 29.4.)
#pragma once
#include "layer_tc_kernel.cuh"

namespace lawcat {
namespace tc {
namespace st {

constexpr int THREADS = 256;
constexpr uint32_t OFF_W = 0;                    // W_h^T fp16: row = output channel, K-major, slabs of 64 channels [128 x 128 B]
constexpr uint32_t OFF_RAW = OFF_W + 32768;      // raw key rows bf16, slabs [64 x 128 B]
constexpr uint32_t OFF_U = OFF_RAW + 16384;      // conv output fp16, the same layout: K-major B of the mix
constexpr uint32_t OFF_G = OFF_U + 16384;        // gate logits bf16, slabs [64 x 128 B]
constexpr uint32_t OFF_V = OFF_G + 16384;        // v bf16, then fp16 in place: MN-major B of the state update
constexpr uint32_t OFF_TAPS = OFF_V + 16384;     // taps as packed pairs: 16-byte unit (2 channel pair + tap / 2) of octet o at (unit * 16 + o) * 16
constexpr uint32_t OFF_HALO = OFF_TAPS + 2048;   // [2 parities][3 rows][16 x 16 B]
constexpr uint32_t OFF_TOT = OFF_HALO + 1536;    // [2 halves][128] log2-decay of half a chunk
constexpr uint32_t OFF_MAX = OFF_TOT + 1024;     // [2 heads][64] row max times log2(e), where it is needed
constexpr uint32_t OFF_SUM = OFF_MAX + 512;      // [4 channel warps][64 tokens] partial softmax sums; the end: z of [2 halves][128]
constexpr uint32_t OFF_INV = OFF_SUM + 1024;     // [8 warps][32 tokens] 1 / sum
constexpr uint32_t OFF_G1 = OFF_INV + 1024;      // [64] log-decays of one decay per head
constexpr uint32_t OFF_BAR = OFF_G1 + 256;
constexpr uint32_t SMEM_BYTES = OFF_BAR + 64;
static_assert(SMEM_BYTES <= 115000, "two blocks per SM");
constexpr uint32_t COL_Y = 0, COL_KH = 64, COL_S = 128, TMEM_COLS = 256;
// (exp(24) is far from any limit. The rounding of y log2(e) is up to 2^-19 at 24, 2^-22 at 4: a feature is off by up to 1.3e-6 or 3e-7
// of itself before it is rounded to fp16, 2.4e-4. End states against 64 bits: the same to four digits as with the maximum taken off.)
constexpr float Y_MAX = 24.f;
enum { B_RAW = 0, B_G, B_V, B_MIX, B_UPD, NUM_BARS };

// one value in all lanes: the largest (NaN counts as nothing)
__device__ __forceinline__ float redux_max(float v) {
  float r;
  asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(v));
  return r;
}
// D (+)= A B with A in tensor memory (lanes = rows, two consecutive K entries per column)
__device__ __forceinline__ void mma_f16_ta(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
      ::"r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}
__device__ __forceinline__ void tmem_st16u(uint32_t taddr, const uint32_t* v) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
      "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
      ::"r"(taddr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "r"(v[8]), "r"(v[9]),
        "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15])
      : "memory");
}

// WIDTH as in the layer kernel: 0 = a head of 128 channels; 1 = one head of 64 (lanes 64-127 idle); 2 = two heads of 64 of one
// key/value group (lanes 0-63, 64-127).
template <int WIDTH>
__global__ void __launch_bounds__(THREADS, 2)
layer_state_kernel(const __grid_constant__ CUtensorMap tm_k, const __grid_constant__ CUtensorMap tm_v,
                   const __grid_constant__ CUtensorMap tm_g, const TcArgs a, const __grid_constant__ PackTab tab) {
  extern __shared__ __align__(1024) uint8_t sg[];
  const uint32_t sb = smem_u32(sg);
  volatile int* const s_flags = reinterpret_cast<volatile int*>(sg + OFF_BAR + 8 * NUM_BARS);  // [0] tmem base, [1] abort
  volatile int* const s_abort = s_flags + 1;
  auto bar = [&](int i) -> uint32_t { return sb + OFF_BAR + 8 * i; };
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;  // (warp: uniform to the compiler)
  constexpr bool narrow = WIDTH == 1, pair = WIDTH == 2, wide = WIDTH == 0;
  constexpr int hd = wide ? 128 : 64, slabs = hd >> 6;  // width of a head; slabs of k and v
  constexpr int gslabs = narrow ? 1 : 2;                // slabs of the gate tile (pair: 128 channels of two heads)
  const int Hn = pair ? a.H / 2 : a.H;
  int blk = blockIdx.x;
  const SeqView sq = seq_of_block(a, tab, Hn * a.nsub, 1, blk);
  const int segs_run = sq.nseg - 1;
  const int sub = blk % a.nsub, seg = (blk / a.nsub) % segs_run, h = blk / (a.nsub * segs_run), b = sq.seq;
  const int h0 = pair ? 2 * h : h, j = h0 / (a.H / a.Hkv);
  const int cps = sq.seg_len / C;
  // (only whole chunks: the ragged end of a sequence lies in its last segment)
  const int t_begin = seg * sq.seg_len + (sub * cps / a.nsub) * C, nchunks = (sub + 1) * cps / a.nsub - sub * cps / a.nsub;
  const size_t out_idx = ((size_t)(sq.seg0 + seg) * a.nsub + sub) * a.H + h0;  // (pair: the second head follows)
  if ((sb & 1023u) != 0) {
    if (tid == 0 && a.dev_status) atomicMax(a.dev_status, (int)LAWCAT_ERR_CUDA);
    return;
  }
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");  // (the scan may be scheduled behind)
  asm volatile("griddepcontrol.wait;" ::: "memory");

  const int tt_first = sq.tm_t + t_begin;
  auto load_raw = [&](int n) {
    mbar_arrive_expect_tx(bar(B_RAW), 8192u * (uint32_t)slabs);
    for (int s = 0; s < slabs; ++s) tma_load_4d(sb + OFF_RAW + s * 8192, &tm_k, bar(B_RAW), s * 64, j, tt_first + n * C, sq.tm_b);
  };
  auto load_gate = [&](int n) {
    mbar_arrive_expect_tx(bar(B_G), 8192u * (uint32_t)gslabs);
    for (int s = 0; s < gslabs; ++s) tma_load_4d(sb + OFF_G + s * 8192, &tm_g, bar(B_G), s * 64, h, tt_first + n * C, sq.tm_b);
  };
  auto load_v = [&](int n) {
    mbar_arrive_expect_tx(bar(B_V), 8192u * (uint32_t)slabs);
    for (int s = 0; s < slabs; ++s) tma_load_4d(sb + OFF_V + s * 8192, &tm_v, bar(B_V), s * 64, j, tt_first + n * C, sq.tm_b);
  };
  // last chunk whose copies / products were issued (first thread)
  int is_raw = -1, is_g = -1, is_v = -1, is_mix = -1, is_upd = -1;
  if (tid == 0) {
    for (int i = 0; i < NUM_BARS; ++i) mbar_init(bar(i), 1);
    mbar_fence_init();
    s_flags[1] = 0;
    if (nchunks > 0) {
      load_raw(0); is_raw = 0;
      if (a.gate_dim != 1) { load_gate(0); is_g = 0; }
      load_v(0); is_v = 0;
    }
  }
  if (warp == 1) {
    tmem_alloc(sb + OFF_BAR + 8 * NUM_BARS, TMEM_COLS);
    tmem_relinquish();
  }
  // raw rows in front of the piece: earlier tokens, or the conv cache, or zeros (Section 4.1)
  constexpr int OCT = hd / 8;
  if (tid >= 64 && tid < 64 + 3 * OCT) {
    const int hr = (tid - 64) / OCT, oc = (tid - 64) % OCT;
    const size_t rstride = (size_t)a.Hkv * hd, coff = (size_t)j * hd + oc * 8;
    const int t = t_begin - HALO + hr, ci = t + (a.K - 1);
    uint4 v = make_uint4(0u, 0u, 0u, 0u);
    if (t >= 0) v = *reinterpret_cast<const uint4*>(a.k + (sq.row0 + t) * rstride + coff);
    else if (a.cache_k && ci >= 0) v = *reinterpret_cast<const uint4*>(a.cache_k + ((size_t)b * (a.K - 1) + ci) * rstride + coff);
    *reinterpret_cast<uint4*>(sg + OFF_HALO + (hr * 16 + oc) * 16) = v;
  }
  for (int i = tid; i < OCT * 16; i += THREADS) {  // octet i % OCT, channel pair and tap i / OCT
    const int o = i % OCT, cp = i / OCT >> 2, dl = i / OCT & 3;
    const bf16* w = a.w_k + ((size_t)j * hd + o * 8 + 2 * cp) * a.K + dl;
    const uint64_t t = dl < a.K ? f2_pack(__bfloat162float(w[0]), __bfloat162float(w[a.K])) : f2_pack(0.f, 0.f);
    *reinterpret_cast<uint64_t*>(sg + OFF_TAPS + ((2 * cp + (dl >> 1)) * 16 + o) * 16 + (dl & 1) * 8) = t;
  }
  // W_h^T: a thread takes channels 2 lane, 2 lane + 1 of a slab and eight output channels (pair: rows 64-127 are the second
  // head's; narrow: they stay as they are, and so nothing in lanes 64-127 means anything)
  {
    constexpr int NI = wide ? 32 : pair ? 16 : 8;  // (octet of outputs, slab)
#pragma unroll
    for (int it = warp; it < NI; it += 8) {
      const int oct = it & 15, slab = it >> 4;
      const bf16* Wc = a.W + ((size_t)(h0 + (pair ? oct >> 3 : 0)) * hd + slab * 64 + 2 * lane) * hd + (pair ? oct & 7 : oct) * 8;
      float x[8], y[8];
      unpack8(*reinterpret_cast<const uint4*>(Wc), x);
      unpack8(*reinterpret_cast<const uint4*>(Wc + hd), y);
#pragma unroll
      for (int i = 0; i < 8; ++i)
        *reinterpret_cast<uint32_t*>(sg + OFF_W + slab * 16384 + sw128(oct * 8 + i, lane >> 2) + (lane & 3) * 4) = pack_f16(x[i], y[i]);
    }
  }
  fence_proxy_async();
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem = (uint32_t)s_flags[0];
  const uint32_t lane_base = tmem + ((uint32_t)((warp & 3) * 32) << 16);
  const int c = (warp & 3) * 32 + lane, th = warp >> 2;  // this thread's channel, its half of the tokens / of the state's columns
  const bool on = !narrow || (warp & 3) < 2;             // (warp-uniform) the channel exists
  const int grp = pair ? (warp & 3) >> 1 : 0;
  float* const s_tot = reinterpret_cast<float*>(sg + OFF_TOT);
  float* const s_sum = reinterpret_cast<float*>(sg + OFF_SUM);
  float* const s_inv = reinterpret_cast<float*>(sg + OFF_INV);
  float* const s_g1 = reinterpret_cast<float*>(sg + OFF_G1);
  const float L2E = 1.4426950408889634f;
  auto wait = [&](int i, int n) { if (!*s_abort) wait_or_abort(bar(i), (uint32_t)(n & 1), s_abort, a.wait_limit); };

  // conv of chunk n: raw rows -> fp16 operand; thread = (octet, run of rows). The halo of the next chunk goes to the other parity.
  auto conv = [&](int n) {
    constexpr int RPT = C * OCT / THREADS;
    const int o = tid % OCT, r0 = tid / OCT * RPT, p = n & 1;
    const uint32_t src = sb + OFF_RAW + (o >> 3) * 8192, dst = sb + OFF_U + (o >> 3) * 8192;
    wait(B_RAW, n);
    uint64_t w[4][4], x0[4], x1[4], x2[4], x3[4];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const uint4 t = lds128(sb + OFF_TAPS + (u * 16 + o) * 16);
      w[u >> 1][2 * (u & 1)] = f2_pack(__uint_as_float(t.x), __uint_as_float(t.y));
      w[u >> 1][2 * (u & 1) + 1] = f2_pack(__uint_as_float(t.z), __uint_as_float(t.w));
    }
    auto row = [&](int r) -> uint4 { return lds128(r < 0 ? sb + OFF_HALO + p * 768 + (r + HALO) * 256 + o * 16 : src + sw128(r, o & 7)); };
    unpack8p(row(r0 - 3), x3); unpack8p(row(r0 - 2), x2); unpack8p(row(r0 - 1), x1);
#pragma unroll
    for (int i = 0; i < RPT; ++i) {
      unpack8p(lds128(src + sw128(r0 + i, o & 7)), x0);
      uint64_t u[4];
#pragma unroll
      for (int cp = 0; cp < 4; ++cp)
        u[cp] = f2_fma(w[cp][0], x0[cp], f2_fma(w[cp][1], x1[cp], f2_fma(w[cp][2], x2[cp], f2_mul(w[cp][3], x3[cp]))));
      sts128(dst + sw128(r0 + i, o & 7), pack8p(u, true));
#pragma unroll
      for (int cp = 0; cp < 4; ++cp) { x3[cp] = x2[cp]; x2[cp] = x1[cp]; x1[cp] = x0[cp]; }
    }
    if (r0 + RPT == C) {
      const uint32_t hl = sb + OFF_HALO + (p ^ 1) * 768 + o * 16;
      sts128(hl, pack8p(x3, false)); sts128(hl + 256, pack8p(x2, false)); sts128(hl + 512, pack8p(x1, false));
    }
  };
  const uint64_t dsc_w = smem_desc(sb + OFF_W, 16, 1024, LAYOUT_SW128), dsc_u = smem_desc(sb + OFF_U, 16, 1024, LAYOUT_SW128);
  const uint64_t dsc_v = smem_desc(sb + OFF_V, 8192, 1024, LAYOUT_SW128);
  auto adv = [](uint64_t d, uint32_t off16) -> uint64_t { return (d & 0xFFFFFFFF00000000ull) | (uint64_t)((uint32_t)d + off16); };
  auto issue_mix = [&](int n) {
    constexpr uint32_t ID = instr_desc(128, C, FMT_F16, MAJOR_K, MAJOR_K);
#pragma unroll
    for (int k = 0; k < hd / 16; ++k)
      mma_f16(tmem + COL_Y, adv(dsc_w, (uint32_t)((k >> 2) * 1024 + (k & 3) * 2)), adv(dsc_u, (uint32_t)((k >> 2) * 512 + (k & 3) * 2)), ID, k > 0);
    mma_commit(bar(B_MIX));
  };
  auto go = [&]() -> bool { return __shfl_sync(0xffffffffu, (int)!*s_abort, 0) != 0; };  // (whole warp)
  auto publish = [&]() {
    fence_proxy_async();
    tc_fence_before_sync();
    __syncthreads();
    tc_fence_after_sync();
  };
  float g1 = 0.f;  // gate_dim = 1: token tid's logit of the next chunk
  auto gate1_load = [&](int n) {
    if (a.gate_dim == 1 && tid < C && n < nchunks) g1 = __bfloat162float(a.gate[(sq.row0 + t_begin + n * C + tid) * a.H + h]);
  };
  gate1_load(0);
  float dsum = 0.f, zacc = 0.f;
  if (nchunks > 0) {
    conv(0);
    publish();
    if (warp == 0 && go()) {
      if (elect_one()) {
        issue_mix(0);
        if (1 < nchunks) load_raw(1);
      }
      is_mix = 0;
      if (1 < nchunks) is_raw = 1;
    }
  }
#pragma unroll 1
  for (int n = 0; n < nchunks; ++n) {
    // ---- gate: x_i = sum of the log2-decays behind token i in this thread's half
    float x[32], tot = 0.f;
    if (a.gate_dim == 1) {
      if (tid < C) s_g1[tid] = a.gate_mode == LAWCAT_GATE_LOGDECAY ? g1 * L2E : log2_sigmoid(g1) * a.inv_tau;
      gate1_load(n + 1);
      __syncthreads();
#pragma unroll
      for (int i = 31; i >= 0; --i) { x[i] = tot; tot += s_g1[th * 32 + i]; }
    } else {
      wait(B_G, n);
      const uint8_t* gcol = sg + OFF_G + (c >> 6) * 8192 + th * 4096 + (c & 7) * 2;
      const int jc = (c & 63) >> 3;
      if (on) {
#pragma unroll
        for (int i = 0; i < 32; ++i) x[i] = __uint_as_float((uint32_t) * reinterpret_cast<const uint16_t*>(gcol + sw128(i, jc)) << 16);
        if (a.gate_mode == LAWCAT_GATE_LOGDECAY) {
#pragma unroll
          for (int i = 31; i >= 0; --i) { const float g = x[i]; x[i] = tot; tot = fmaf(L2E, g, tot); }
        } else {
#pragma unroll
          for (int i = 0; i < 32; i += 2) {  // (log2_sigmoid, two at a time where the instructions come in pairs)
            float l0, l1, s0, s1;
            f2_unpack(f2_mul(f2_pack(x[i], x[i + 1]), f2_pack(-L2E, -L2E)), l0, l1);
            f2_unpack(f2_add(f2_pack(ex2f(fminf(l0, 126.f)), ex2f(fminf(l1, 126.f))), f2_pack(1.f, 1.f)), s0, s1);
            x[i] = fmaxf(l0, lg2f(s0));
            x[i + 1] = fmaxf(l1, lg2f(s1));
          }
#pragma unroll
          for (int i = 31; i >= 0; --i) { const float g = x[i]; x[i] = tot; tot = fmaf(-a.inv_tau, g, tot); }
        }
      }
    }
    s_tot[th * 128 + c] = tot;
    if (tid == 0 && n > 0 && !*s_abort) {  // v behind the product that read the chunk in front's (it has completed by now)
      wait(B_UPD, n - 1);
      if (!*s_abort) { load_v(n); is_v = n; }
    }
    // ---- features: softmax over the channels of a token. While every |y| stays below Y_MAX, exp(y) needs no shift by the row's
    // maximum: the sums are formed without waiting for it, and the barrier that makes them known also tells whether one is missing.
    wait(B_MIX, n);
    tc_fence_after_sync();
    float y[32];
    auto sums = [&]() {  // over the lanes, every step halving the tokens a lane carries: lane l ends with token l
      float s[16];
      {
        const bool up = lane & 16;
#pragma unroll
        for (int i = 0; i < 16; ++i) s[i] = (up ? y[i + 16] : y[i]) + __shfl_xor_sync(0xffffffffu, up ? y[i] : y[i + 16], 16);
      }
#pragma unroll
      for (int w = 8; w > 0; w >>= 1) {
        const bool up = lane & w;
#pragma unroll
        for (int i = 0; i < 8; ++i)
          if (i < w) s[i] = (up ? s[i + w] : s[i]) + __shfl_xor_sync(0xffffffffu, up ? s[i] : s[i + w], w);
      }
      s_sum[((warp & 3) * 2 + th) * 32 + lane] = s[0];
    };
    bool big = false;
    if (on) {
      tmem_ld32(lane_base + COL_Y + th * 32, y);
      tmem_wait_ld();
      float m = 0.f;
#pragma unroll
      for (int i = 0; i < 32; ++i) m = fmaxf(m, fabsf(y[i]));
      big = !(m < Y_MAX);
#pragma unroll
      for (int i = 0; i < 32; ++i) y[i] = ex2f(y[i] * L2E);
      sums();
    }
    if (__syncthreads_or(big)) {
      float* const s_max = reinterpret_cast<float*>(sg + OFF_MAX) + grp * 64 + th * 32;
      if (tid < 128) reinterpret_cast<float*>(sg + OFF_MAX)[tid] = -INFINITY;
      __syncthreads();
      if (on) {
        tmem_ld32(lane_base + COL_Y + th * 32, y);
        tmem_wait_ld();
        float m = 0.f;
#pragma unroll
        for (int i = 0; i < 32; ++i) {
          const float r = redux_max(y[i]);
          if (lane == i) m = r;
        }
        m = fmaf(m, L2E, 0.f);  // (never -0: the order of the two atomics)
        if (m >= 0.f) atomicMax(reinterpret_cast<int*>(s_max + lane), __float_as_int(m));
        else atomicMin(reinterpret_cast<unsigned*>(s_max + lane), __float_as_uint(m));
      }
      __syncthreads();
      if (on) {
#pragma unroll
        for (int i = 0; i < 32; ++i) y[i] = ex2f(fmaf(y[i], L2E, -s_max[i]));
        sums();
      }
      __syncthreads();
    }
    if (tid == 0 && a.gate_dim != 1 && n + 1 < nchunks && !*s_abort) { load_gate(n + 1); is_g = n + 1; }
    if (on) {  // 1 / sum of this warp's tokens, for its own use
      const float* const t = s_sum + (grp * 4 + th) * 32 + lane;
      s_inv[warp * 32 + lane] = 1.f / (wide ? (t[0] + t[64]) + (t[128] + t[192]) : t[0] + t[64]);
      __syncwarp();
    }
    // ---- state: decay of this thread's columns of its row
    const float tot_all = s_tot[c] + s_tot[128 + c], dC = ex2f(tot_all);
    dsum += tot_all;
    zacc *= dC;
    if (n > 0) {
      wait(B_UPD, n - 1);
      tc_fence_after_sync();
      if (on) {
        const uint64_t d2 = f2_pack(dC, dC);
#pragma unroll 1
        for (int b2 = 0; b2 < (wide ? 2 : 1); ++b2) {
          const uint32_t col = lane_base + COL_S + th * (hd / 2) + b2 * 32;
          float s[32];
          tmem_ld32(col, s);
          tmem_wait_ld();
#pragma unroll
          for (int i = 0; i < 32; i += 2) f2_unpack(f2_mul(d2, f2_pack(s[i], s[i + 1])), s[i], s[i + 1]);
          tmem_st32(col, s);
        }
      }
    }
    // ---- kh_i = phi_i 2^(b_C - b_i), rounded to fp16, into tensor memory
    if (on) {
      const float off = th ? 0.f : s_tot[128 + c];  // the decay of the half behind
      const float* const inv = s_inv + warp * 32;
      const uint64_t off2 = f2_pack(off, off);
      uint64_t zs = 0ull;
      uint32_t kh[16];
#pragma unroll
      for (int q4 = 0; q4 < 8; ++q4) {
        const ulonglong2 iv = *reinterpret_cast<const ulonglong2*>(inv + 4 * q4);
#pragma unroll
        for (int i = 4 * q4; i < 4 * q4 + 4; i += 2) {
          float e0, e1, k0, k1;
          f2_unpack(f2_add(f2_pack(x[i], x[i + 1]), off2), e0, e1);
          const uint64_t k2 = f2_mul(f2_mul(f2_pack(y[i], y[i + 1]), i & 2 ? iv.y : iv.x), f2_pack(ex2f(e0), ex2f(e1)));
          f2_unpack(k2, k0, k1);
          const __half2 h2 = __floats2half2_rn(k0, k1);
          kh[i / 2] = *reinterpret_cast<const uint32_t*>(&h2);
          const float2 kr = __half22float2(h2);  // (z as the layer kernel has it: the sum of the keys AS ROUNDED)
          zs = f2_add(zs, f2_pack(kr.x, kr.y));
        }
      }
      float z0, z1;
      f2_unpack(zs, z0, z1);
      zacc += z0 + z1;
      tmem_st16u(lane_base + COL_KH + th * 16, kh);
      tmem_wait_st();
    }
    if (n + 1 < nchunks) conv(n + 1);
    // ---- v: bf16 -> fp16 in place (exact for |v| in the fp16 normal range)
    wait(B_V, n);
#pragma unroll
    for (int i = 0; i < slabs * 512 / THREADS; ++i) {
      const uint32_t ad = sb + OFF_V + (uint32_t)(tid + THREADS * i) * 16;
      float f[8];
      unpack8(lds128(ad), f);
      sts128(ad, pack8(f, true));
    }
    publish();
    if (warp == 0 && go()) {
      if (elect_one()) {
        constexpr uint32_t ID = instr_desc(128, hd, FMT_F16, MAJOR_K, MAJOR_MN);
#pragma unroll
        for (int k = 0; k < C / 16; ++k)
          mma_f16_ta(tmem + COL_S, tmem + COL_KH + 8 * k, adv(dsc_v, (uint32_t)k * (2048 >> 4)), ID, n > 0 || k > 0);
        mma_commit(bar(B_UPD));
        if (n + 1 < nchunks) issue_mix(n + 1);
        if (n + 2 < nchunks) load_raw(n + 2);
      }
      is_upd = n;
      if (n + 1 < nchunks) is_mix = n + 1;
      if (n + 2 < nchunks) is_raw = n + 2;
    }
  }
  // ---- end state, as whole rows through the dead tiles
  if (nchunks > 0) wait(B_UPD, nchunks - 1);
  tc_fence_after_sync();
  const bool ok = !*s_abort;
  constexpr int UPR = hd / 4;  // 16-byte units per row
  if (on && ok) {
#pragma unroll 1
    for (int b2 = 0; b2 < (wide ? 2 : 1); ++b2) {
      float s[32];
      if (nchunks > 0) {
        tmem_ld32(lane_base + COL_S + th * (hd / 2) + b2 * 32, s);
        tmem_wait_ld();
      } else {
#pragma unroll
        for (int i = 0; i < 32; ++i) s[i] = 0.f;
      }
#pragma unroll
      for (int q4 = 0; q4 < 8; ++q4) {
        const int unit = th * (hd / 8) + b2 * 8 + q4;
        sts128(sb + OFF_RAW + (uint32_t)(c * UPR + (unit ^ (c & 7))) * 16u,
               make_uint4(__float_as_uint(s[4 * q4]), __float_as_uint(s[4 * q4 + 1]), __float_as_uint(s[4 * q4 + 2]), __float_as_uint(s[4 * q4 + 3])));
      }
    }
    s_sum[th * 128 + c] = zacc;
  }
  tc_fence_before_sync();
  __syncthreads();
  if (*s_abort) {
    if (tid == 0) {
      // leaving early: a bounded time for the copies and products still under way
      if (is_raw >= 0) mbar_wait(bar(B_RAW), (uint32_t)(is_raw & 1));
      if (is_g >= 0) mbar_wait(bar(B_G), (uint32_t)(is_g & 1));
      if (is_v >= 0) mbar_wait(bar(B_V), (uint32_t)(is_v & 1));
      if (is_mix >= 0) mbar_wait(bar(B_MIX), (uint32_t)(is_mix & 1));
      if (is_upd >= 0) mbar_wait(bar(B_UPD), (uint32_t)(is_upd & 1));
      if (a.dev_status) atomicMax(a.dev_status, (int)LAWCAT_ERR_TIMEOUT);
    }
    __syncthreads();
  } else {
    constexpr int ROWS = narrow ? 64 : 128;
    float* const dS = a.S_T + out_idx * hd * hd;
#pragma unroll 4
    for (int i = tid; i < ROWS * UPR; i += THREADS) {
      const int r = i / UPR, unit = i % UPR;
      *reinterpret_cast<uint4*>(dS + (size_t)r * hd + unit * 4) = lds128(sb + OFF_RAW + (uint32_t)(r * UPR + (unit ^ (r & 7))) * 16u);
    }
    if (tid < ROWS) {
      a.z_T[out_idx * hd + tid] = s_sum[tid] + s_sum[128 + tid];
    }
    if (on && th == 0) a.dtot[out_idx * hd + c] = dsum;
  }
  if (warp == 1) {
    tc_fence_after_sync();
    tmem_dealloc(tmem, TMEM_COLS);
  }
}

}  // namespace st
}  // namespace tc
}  // namespace lawcat
