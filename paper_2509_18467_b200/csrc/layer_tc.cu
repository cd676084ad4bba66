// Host side of the chunkwise tensor-core layer forward: tensor maps, segment split, launches.
#include <algorithm>
#include <atomic>
#include <mutex>
#include <vector>

#include "layer_state_kernel.cuh"
#include "layer_tc_kernel.cuh"

namespace lawcat {
namespace tc {

// ---------------------------------------------------------------------------------------------------- host side
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                  const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      p = nullptr;
    return (EncodeTiledFn)p;
  }();
  return fn;
}

}  // namespace tc

// A map depends only on the pointer and the shape, so the last few are kept per host thread: a serving loop that calls
// with the same buffers encodes each map once.
bool tensor_map(CUtensorMap* m, const void* ptr, bool f32, int heads, int T, int B, int dh, int box_ch, int rows, bool swizzle) {
  struct Slot {
    const void* ptr;
    int heads, T, B, dh, box_ch, rows;
    bool f32, swizzle, used;
    CUtensorMap map;
  };
  constexpr int NSLOT = 32;
  thread_local Slot cache[NSLOT] = {};
  thread_local int next = 0;
  for (int i = 0; i < NSLOT; ++i) {
    const Slot& c = cache[i];
    if (c.used && c.ptr == ptr && c.heads == heads && c.T == T && c.B == B && c.dh == dh && c.box_ch == box_ch && c.rows == rows &&
        c.f32 == f32 && c.swizzle == swizzle) {
      *m = c.map;
      return true;
    }
  }
  tc::EncodeTiledFn fn = tc::encode_fn();
  if (!fn) return false;
  const cuuint64_t row = (cuuint64_t)dh * (f32 ? 4 : 2);
  const cuuint64_t dims[4] = {(cuuint64_t)dh, (cuuint64_t)heads, (cuuint64_t)T, (cuuint64_t)B};
  const cuuint64_t strides[3] = {row, heads * row, T * (heads * row)};
  const cuuint32_t box[4] = {(cuuint32_t)box_ch, 1, (cuuint32_t)rows, 1};
  const cuuint32_t es[4] = {1, 1, 1, 1};
  if (fn(m, f32 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(ptr), dims, strides, box, es,
         CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_NONE,
         CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
    return false;
  Slot& c = cache[next];
  next = (next + 1) % NSLOT;
  c.ptr = ptr; c.heads = heads; c.T = T; c.B = B; c.dh = dh; c.box_ch = box_ch; c.rows = rows; c.f32 = f32; c.swizzle = swizzle;
  c.map = *m; c.used = true;
  return true;
}

namespace tc {

// [B, T, heads, dh] bf16 tensor in boxes of 64 channels x rows tokens, 128-byte-swizzled
static bool make_map(CUtensorMap* m, const void* ptr, int heads, int T, int B, int rows, int dh) {
  return tensor_map(m, ptr, false, heads, T, B, dh, 64, rows, true);
}

// State at the start of every segment but a sequence's first from the end states of the pieces in front (each computed from a
// zero state) and their total decays: running state cur = given state; after piece i: cur = decay[i] * cur + local[i] (Eq. 4
// unrolled over whole pieces). One thread per four state entries (the d_k x d_v entries of S, then the d_k entries of z) of one
// (sequence, head).
__global__ void segment_scan_kernel(const TcArgs a, const __grid_constant__ PackTab tab, const float* __restrict__ loc_S,
                                    const float* __restrict__ loc_z, const float* __restrict__ dtot, float* __restrict__ start_S,
                                    float* __restrict__ start_z, int nseq, int nsub, int dh) {
  const int D = dh;  // (rows and columns of the state as stored)
  const int per = (D * D + D) / 4;
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  asm volatile("griddepcontrol.wait;" ::: "memory");               // behind the state-only pass
  if (idx >= nseq * a.H * per) return;
  const int e = idx % per * 4, h = idx / per % a.H;
  const int i = idx / (per * a.H);
  const int seg0 = tab.n ? tab.seg0[i] : i * a.nseg, nseg = tab.n ? tab.seg0[i + 1] - seg0 : a.nseg;
  const int seq = tab.n ? tab.seq[i] : i;
  const bool isz = e >= D * D;
  const float* const init = isz ? a.z0 : a.S0;
  const size_t n = isz ? D : (size_t)D * D, off = isz ? e - D * D : e;  // entries per state, this thread's first
  const float* const loc = isz ? loc_z : loc_S;
  float* const start = isz ? start_z : start_S;
  float4 cur = make_float4(0.f, 0.f, 0.f, 0.f);
  if (init) cur = *reinterpret_cast<const float4*>(init + ((size_t)seq * a.H + h) * n + off);
  // With few heads the blocks are few and a thread's own instructions are the time: the loop walks pointers and a counter
  // of the pieces left in the segment, and the decay of a row of S is one exponential.
  const int np = (nseg - 1) * nsub;
  const size_t lstep = (size_t)a.H * n, dstep = (size_t)a.H * D;
  const float* lp = loc + ((size_t)seg0 * nsub * a.H + h) * n + off;
  const float* dp = dtot + ((size_t)seg0 * nsub * a.H + h) * D + (isz ? off : off / D);
  float* sp = start + ((size_t)(seg0 + 1) * a.H + h) * n + off;
  int left = nsub;
  auto batch = [&](auto count) {  // pieces whose loads are in flight together
    constexpr int U = decltype(count)::value;
    float4 l[U], d[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      l[u] = *reinterpret_cast<const float4*>(lp + u * lstep);
      if (isz) d[u] = *reinterpret_cast<const float4*>(dp + u * dstep);
      else d[u].x = dp[u * dstep];
    }
    lp += U * lstep;
    dp += U * dstep;
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const float ex = exp2f(d[u].x);
      float4 e = make_float4(ex, ex, ex, ex);
      if (isz) e = make_float4(ex, exp2f(d[u].y), exp2f(d[u].z), exp2f(d[u].w));
      cur.x = fmaf(e.x, cur.x, l[u].x); cur.y = fmaf(e.y, cur.y, l[u].y);
      cur.z = fmaf(e.z, cur.z, l[u].z); cur.w = fmaf(e.w, cur.w, l[u].w);
      if (--left == 0) {
        left = nsub;
        *reinterpret_cast<float4*>(sp) = cur;
        sp += lstep;
      }
    }
  };
  int i0 = 0;
  for (; i0 + 8 <= np; i0 += 8) batch(std::integral_constant<int, 8>{});
  if (i0 + 4 <= np) { batch(std::integral_constant<int, 4>{}); i0 += 4; }
  if (np - i0 == 3) batch(std::integral_constant<int, 3>{});
  else if (np - i0 == 2) batch(std::integral_constant<int, 2>{});
  else if (np - i0 == 1) batch(std::integral_constant<int, 1>{});
}

}  // namespace tc

// Number of SMs of the current device (cached per device; 148 on a B200).
int sm_count() {
  static int cached[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 148;
  if (cached[dev] == 0) {
    int n = 0;
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) n = 148;
    cached[dev] = n;
  }
  return cached[dev];
}

// How a sequence is cut: nseg segments of seg_len tokens (a multiple of the chunk; every segment holds tokens), and the
// pieces per segment of the state-only pre-pass.
struct TcPlan {
  int nseg, seg_len, nsub;
};

// Segments per sequence: enough thread blocks to fill the SMs (one block per SM), but at least MIN_SEG_CHUNKS chunks per
// segment (a thread block spends about three chunk times on its set-up and on filling its pipeline). Pieces per segment
// in the state-only pre-pass: its thread blocks are independent, so cutting the segments finer lets them fill the SMs, two to
// an SM, in whole waves; the split with the fewest chunks per SM wins (a set-up is two chunk times). Measured over 1 to 8 pieces:
// 32768 tokens, 32 heads of 128: 460 us as one piece, 337, 232 as three (96 blocks each), 275 as four, 237 as six; 1223 tokens
// (five chunks a segment): the call 66.6 us, 67.8, 64.6 as three, 73.8 as four.
// Two 64-wide heads share a thread block when they can: an even number of query heads per key/value head (the two heads
// of a block read the same k and v) and one decay per key channel.
static bool layer_tc_paired(const lawcat_params& p) {
  return p.d_k == 64 && p.gate_dim == p.d_k && (p.H / p.H_kv) % 2 == 0;
}

static TcPlan layer_tc_plan(const lawcat_params& p) {
  constexpr int MIN_SEG_CHUNKS = 4;
  const int sms = sm_count();
  const int chunks = (p.T + tc::C - 1) / tc::C;
  const int seqs = p.B * (layer_tc_paired(p) ? p.H / 2 : p.H);  // sequences of thread blocks
  int n = sms / seqs;
  if (n > chunks / MIN_SEG_CHUNKS) n = chunks / MIN_SEG_CHUNKS;
  if (n < 1) n = 1;
  TcPlan pl;
  pl.seg_len = ((chunks + n - 1) / n) * tc::C;
  pl.nseg = (p.T + pl.seg_len - 1) / pl.seg_len;  // (rounding the length up may leave fewer segments than asked for)
  if (pl.nseg < 1) pl.nseg = 1;
  const int cps = pl.seg_len / tc::C;
  int best = 1, best_cost = 1 << 30;
  for (int ns = 1; ns <= 8 && ns * 2 <= cps + 1; ++ns) {
    const int ctas = seqs * (pl.nseg - 1) * ns;
    const int cost = ((ctas + 2 * sms - 1) / (2 * sms)) * ((cps + ns - 1) / ns + 2);
    if (cost < best_cost) { best_cost = cost; best = ns; }
  }
  pl.nsub = best;
  return pl;
}

// Limit of the kernels' device-side waits in clock cycles (about two seconds); a test hook may shorten it.
static std::atomic<long long> g_wait_limit{4000000000LL};
long long wait_limit() { return g_wait_limit.load(); }

// scratch of a launch with `segs` segments in all (none when every sequence is one segment)
static size_t layer_tc_scratch(const lawcat_params& p, size_t segs, int nsub) {
  const size_t pieces = segs * nsub;
  return sizeof(float) * (size_t)p.H * ((pieces + segs) * ((size_t)p.d_k * p.d_k + p.d_k) + pieces * p.d_k);
}

size_t layer_tc_workspace_bytes(const lawcat_params& p) {
  const TcPlan pl = layer_tc_plan(p);
  return pl.nseg == 1 ? 0 : layer_tc_scratch(p, (size_t)p.B * pl.nseg, pl.nsub);
}

// Packed sequences: how one launch cuts them. All sequences of the group share the SMs, so the segments are only as short as
// it takes to keep the longest from being the tail: L, the longest segment allowed, is the one with the smallest estimate of
// chunk times over {longest / 1 .. longest / 8}: per block its chunks and about three more for set-up and pipeline fill, the
// total spread over the SMs but never less than the longest block and half a block of unevenness; when something is cut, the
// state-only pass over all but the last segments and its two extra launches (about two). The pass is charged 0.65 of a chunk time a
// chunk, one block per SM, in pieces of at least four chunks, which is dearer than it is (0.44, two blocks per SM; the price is of the
// time when it was a mode of the layer kernel). The surplus stands in for what the estimate of the main launch leaves out, a last
// round of a few blocks: at the true price 2 sequences of together 2500 tokens, 32 heads of 128, are cut into 160 blocks and take 122 us,
// not 103. Over 70 batches of 2 to 32 sequences this rule is 3.6 % behind the best cut and piece count on average, 28 % at most.
static void layer_tc_pack(const lawcat_params& p, const int32_t* cu, const int* order, int n, tc::PackTab& t, int& nsub) {
  const double sms = sm_count(), Hn = layer_tc_paired(p) ? p.H / 2 : p.H;
  auto chunks = [&](int i) { return (cu[order[i] + 1] - cu[order[i]] + tc::C - 1) / tc::C; };
  const int longest = chunks(0);
  int best_L = longest, best_sub = 1;
  double best = 1e30;
  for (int k = 1; k <= 8 && (k == 1 || longest / k >= 4); ++k) {
    const int L = (longest + k - 1) / k;
    double work = 0, pre = 0, pieces = 0;
    int seg_max = 0;
    for (int i = 0; i < n; ++i) {
      const int ch = chunks(i), ns = (ch + L - 1) / L, sl = (ch + ns - 1) / ns;
      work += ch + 3.0 * ns;
      pre += (double)(ns - 1) * sl;
      pieces += ns - 1;
      if (sl > seg_max) seg_max = sl;
    }
    auto span = [&](double total, double one) { return total * Hn / sms > one ? total * Hn / sms + 0.5 * one : one; };
    const double main_cost = span(work, seg_max + 3.0);
    if (pieces == 0) {
      if (main_cost < best) { best = main_cost; best_L = L; best_sub = 1; }
      continue;
    }
    for (int sub = 1; sub <= 4 && sub * 4 <= seg_max; ++sub) {
      const double cost = main_cost + 2.0 + span(0.65 * (pre + 2.0 * sub * pieces), 0.65 * ((double)seg_max / sub + 2.0));
      if (cost < best) { best = cost; best_L = L; best_sub = sub; }
    }
  }
  nsub = best_sub;
  t.n = n;
  t.seg0[0] = 0;
  for (int i = 0; i < n; ++i) {
    const int ch = chunks(i), ns = (ch + best_L - 1) / best_L, sl = (ch + ns - 1) / ns;
    t.tok0[i] = cu[order[i]];
    t.len[i] = cu[order[i] + 1] - cu[order[i]];
    t.seg_len[i] = sl * tc::C;
    t.seg0[i + 1] = t.seg0[i] + (ch + sl - 1) / sl;
    t.seq[i] = order[i];
  }
}

// the sequences that the packed launches take (those the layer kernel serves: at least 16 tokens), the longest first
static std::vector<int> layer_tc_pack_order(const lawcat_params& p, const int32_t* cu, int nseq) {
  std::vector<int> order;
  lawcat_params q = p;
  q.B = 1;
  for (int i = 0; i < nseq; ++i) {
    q.T = cu[i + 1] - cu[i];
    if (layer_tc_supported(q)) order.push_back(i);
  }
  std::stable_sort(order.begin(), order.end(), [&](int x, int y) { return cu[x + 1] - cu[x] > cu[y + 1] - cu[y]; });
  return order;
}

size_t layer_tc_packed_workspace_bytes(const lawcat_params& p, const int32_t* cu, int nseq) {
  const std::vector<int> order = layer_tc_pack_order(p, cu, nseq);
  size_t need = 0;
  for (size_t o = 0; o < order.size(); o += tc::PACK_MAX) {
    const int n = (int)(order.size() - o < tc::PACK_MAX ? order.size() - o : tc::PACK_MAX);
    tc::PackTab t;
    int nsub = 1;
    layer_tc_pack(p, cu, order.data() + o, n, t, nsub);
    const size_t b = t.seg0[n] == n ? 0 : layer_tc_scratch(p, (size_t)t.seg0[n], nsub);
    if (b > need) need = b;
  }
  return need;
}

bool layer_tc_supported(const lawcat_params& p) {
  // Sharp sigmoid gates (tau < 8: a token's decay reaches a half at tau = 1) drive the exponents of the in-chunk
  // factorization out of the fp16 range within half a chunk; the operands then fall back to bf16 (8 significant bits)
  // and a seeded random sweep finds outputs and states beyond 1e-2 of their RMS for tau = 1, 2 and 4 (numerator-only
  // form, one decay per head, eps != 0, carried states). Those gates take the exact recurrence. Very short calls do too:
  // with fewer than 16 tokens the state is a sum of so few terms that the rounding of single 16-bit operands shows in
  // its largest entries, and the exact kernels are as fast there.
  const bool sharp = p.gate_mode == LAWCAT_GATE_LOGITS && p.gate_tau < 8.f;
  return p.dtype == LAWCAT_BF16 && (p.d_k == tc::D || p.d_k == 64) && p.d_v == p.d_k &&
         (p.gate_dim == p.d_k || p.gate_dim == 1) && !sharp && p.T >= 16 &&
         p.phi == LAWCAT_PHI_SOFTMAX && p.conv_k <= tc::HALO + 1 && p.B > 0 && p.T > 0 &&
         (p.chunk == 0 || p.chunk == tc::C) &&
         !p.mix_unshared;  // (one W_h is what lets both streams share the M = 128 mix)
}

// One launch set over a uniform batch (tab.n = 0) or a group of packed sequences; `segs` segments in all, of `nseq` sequences.
static int run_layer_tc(const Ctx& c, const void* q, const void* k, const void* v, const void* gate, const void* w_q,
                        const void* w_k, const void* W, const void* cache_q_in, const void* cache_k_in, const float* S0,
                        const float* z0, void* o, void* cache_q_out, void* cache_k_out, float* S_T, float* z_T, void* ws,
                        const TcPlan& pl, const tc::PackTab& tab, int nseq, int segs) {
  using namespace tc;
  const lawcat_params& p = *c.p;
  CUtensorMap tq, tk, tv, tg;
  const int dh = p.d_k;
  const bool paired = layer_tc_paired(p);
  // (pair: q, gate and o of two neighbouring heads are 128 contiguous channels and are mapped as one head of 128)
  const int Hmap = paired ? p.H / 2 : p.H, dmap = paired ? 128 : dh;
  if (!make_map(&tq, q, Hmap, p.T, p.B, C, dmap) || !make_map(&tk, k, p.H_kv, p.T, p.B, C, dh) ||
      !make_map(&tv, v, p.H_kv, p.T, p.B, C, dh))
    return LAWCAT_ERR_CUDA;
  if (p.gate_dim == 1) tg = tq;  // (never used: one logit per token and head is read without a tensor map)
  else if (!make_map(&tg, gate, Hmap, p.T, p.B, C, dmap)) return LAWCAT_ERR_CUDA;
  TcArgs a{};
  a.q = (const bf16*)q; a.k = (const bf16*)k; a.o = (bf16*)o;
  a.gate = (const bf16*)gate; a.gate_dim = p.gate_dim; a.dh = dh;
  a.w_q = (const bf16*)w_q; a.w_k = (const bf16*)w_k; a.W = (const bf16*)W;
  a.cache_q = (const bf16*)cache_q_in; a.cache_k = (const bf16*)cache_k_in;
  a.cache_q_out = (bf16*)cache_q_out; a.cache_k_out = (bf16*)cache_k_out;
  a.dev_status = c.dev_status;
  a.T = p.T; a.H = p.H; a.Hkv = p.H_kv; a.K = p.conv_k;
  a.gate_mode = p.gate_mode; a.normalize = p.normalize; a.inv_tau = 1.f / p.gate_tau; a.eps = p.eps;
  a.wait_limit = wait_limit();
  const int nsub = pl.nsub;
  a.nseg = pl.nseg;
  a.seg_len = pl.seg_len;
  a.nsub = 1;
  a.S0 = S0; a.z0 = z0; a.S_T = S_T; a.z_T = z_T;
  auto* const k_layer = paired ? layer_tc_kernel<2> : dh == 64 ? layer_tc_kernel<1> : layer_tc_kernel<0>;
  auto* const k_state = paired ? st::layer_state_kernel<2> : dh == 64 ? st::layer_state_kernel<1> : st::layer_state_kernel<0>;
  {
    // the kernels' shared-memory limit is raised once per device
    static std::mutex mu;
    static bool done[64] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return LAWCAT_ERR_CUDA;
    std::lock_guard<std::mutex> lk(mu);
    if (!done[dev]) {
      if (cudaFuncSetAttribute(layer_tc_kernel<0>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM_ALLOC) != cudaSuccess ||
          cudaFuncSetAttribute(layer_tc_kernel<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM_ALLOC) != cudaSuccess ||
          cudaFuncSetAttribute(layer_tc_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM_ALLOC) != cudaSuccess ||
          cudaFuncSetAttribute(st::layer_state_kernel<0>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)st::SMEM_BYTES) != cudaSuccess ||
          cudaFuncSetAttribute(st::layer_state_kernel<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)st::SMEM_BYTES) != cudaSuccess ||
          cudaFuncSetAttribute(st::layer_state_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)st::SMEM_BYTES) != cudaSuccess)
        return LAWCAT_ERR_CUDA;
      done[dev] = true;
    }
  }
  const int Hn = paired ? p.H / 2 : p.H;          // thread blocks per segment
  if (segs == nseq) {
    LaunchScope _ls("layer_tc", c.stream);
    launch_behind(k_layer, dim3(Hn * segs), dim3(LAYER_THREADS), SMEM_ALLOC, c.stream, tq, tk, tv, tg, a, tab);
    LAWCAT_CHECK_LAUNCH();
    return LAWCAT_OK;
  }
  // Several segments per sequence: (1) every segment but a sequence's last computes its end state from a zero state, and the
  // total decay of the segment; (2) a scan over the segments turns these into the state at each segment's start;
  // (3) the layer runs on all segments at once, each from its start state.
  const size_t nS = (size_t)p.H * segs * dh * dh, nz = (size_t)p.H * segs * dh;
  float* loc_S = (float*)ws;              // [segs, nsub, H, D, D]
  float* loc_z = loc_S + nS * nsub;       // [segs, nsub, H, D]
  float* dtot = loc_z + nz * nsub;        // [segs, nsub, H, D]
  float* start_S = dtot + nz * nsub;      // [segs, H, D, D]
  float* start_z = start_S + nS;          // [segs, H, D]
  {
    TcArgs b1 = a;
    b1.S_T = loc_S; b1.z_T = loc_z; b1.dtot = dtot; b1.nsub = nsub;
    LaunchScope _ls("layer_tc_state", c.stream);
    launch_behind(k_state, dim3(Hn * (segs - nseq) * nsub), dim3(st::THREADS), st::SMEM_BYTES, c.stream, tk, tv, tg, b1, tab);
    LAWCAT_CHECK_LAUNCH();
  }
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.stream = c.stream;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  {
    const int total = nseq * p.H * (dh * dh + dh) / 4;
    LaunchScope _ls("segment_scan", c.stream);
    cfg.gridDim = dim3((unsigned)((total + 127) / 128));
    cfg.blockDim = dim3(128);
    cudaLaunchKernelEx(&cfg, segment_scan_kernel, a, tab, (const float*)loc_S, (const float*)loc_z, (const float*)dtot,
                       start_S, start_z, nseq, nsub, dh);
    LAWCAT_CHECK_LAUNCH();
  }
  a.seg_S = start_S; a.seg_z = start_z;
  {
    // (the scan gives no early start: with one, blocks land while scan blocks still hold registers of most SMs,
    // and the call at T = 32768 took 1.34 ms instead of 1.11)
    LaunchScope _ls("layer_tc", c.stream);
    launch_behind(k_layer, dim3(Hn * segs), dim3(LAYER_THREADS), SMEM_ALLOC, c.stream, tq, tk, tv, tg, a, tab);
  }
  LAWCAT_CHECK_LAUNCH();
  return LAWCAT_OK;
}

int launch_layer_tc(const Ctx& c, const void* q, const void* k, const void* v, const void* gate, const void* w_q,
                    const void* w_k, const void* W, const void* cache_q_in, const void* cache_k_in, const float* S0,
                    const float* z0, void* o, void* cache_q_out, void* cache_k_out, float* S_T, float* z_T, void* ws) {
  const TcPlan pl = layer_tc_plan(*c.p);
  tc::PackTab tab;
  tab.n = 0;
  return run_layer_tc(c, q, k, v, gate, w_q, w_k, W, cache_q_in, cache_k_in, S0, z0, o, cache_q_out, cache_k_out, S_T, z_T, ws,
                      pl, tab, c.p->B, c.p->B * pl.nseg);
}

int launch_layer_tc_packed(const Ctx& c, const int32_t* cu, int nseq, const void* q, const void* k, const void* v,
                           const void* gate, const void* w_q, const void* w_k, const void* W, const void* cache_q_in,
                           const void* cache_k_in, const float* S0, const float* z0, void* o, void* cache_q_out,
                           void* cache_k_out, float* S_T, float* z_T, void* ws) {
  const std::vector<int> order = layer_tc_pack_order(*c.p, cu, nseq);
  for (size_t at = 0; at < order.size(); at += tc::PACK_MAX) {
    const int n = (int)(order.size() - at < tc::PACK_MAX ? order.size() - at : tc::PACK_MAX);
    tc::PackTab tab;
    TcPlan pl{};
    layer_tc_pack(*c.p, cu, order.data() + at, n, tab, pl.nsub);
    const int r = run_layer_tc(c, q, k, v, gate, w_q, w_k, W, cache_q_in, cache_k_in, S0, z0, o, cache_q_out, cache_k_out, S_T,
                               z_T, ws, pl, tab, n, tab.seg0[n]);
    if (r) return r;
  }
  return LAWCAT_OK;
}

}  // namespace lawcat

// Test hook: the limit (clock cycles) of every bounded device-side wait of the layer forward and streaming decode kernels
// launched from now on; 0 restores the default. A limit of a few cycles makes the first unsatisfied wait give up, which exercises the
// path that reports LAWCAT_ERR_TIMEOUT (nothing faults or hangs: the block leaves its loops, lets its copies land, frees
// its tensor memory and returns).
extern "C" void lawcat_test_set_wait_limit(long long cycles) {
  lawcat::g_wait_limit.store(cycles > 0 ? cycles : 4000000000LL);
}

#ifdef LAWCAT_TIMELINE
// (profiling builds only) copies the clock stamps of the last layer-kernel launch to the host
extern "C" int lawcat_timeline_read(long long* host, size_t n) {
  const size_t have = sizeof(lawcat::tc::g_timeline) / sizeof(long long);
  return cudaMemcpyFromSymbol(host, lawcat::tc::g_timeline, sizeof(long long) * (n < have ? n : have)) == cudaSuccess
             ? LAWCAT_OK : LAWCAT_ERR_CUDA;
}
#endif
