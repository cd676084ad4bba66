// Operand tiles of the lock-step tensor-core kernels (conv + mix forward and backward, decode features): unswizzled 8x8
// core matrices with every 8-column slab contiguous. Element (r, c) of a tile with R rows sits at
// (c / 8) * (16 R + 16) + 16 r + 2 (c % 8); the same bytes serve as a K-major operand (LBO = slab stride, SBO = 128) and
// as an MN-major one (LBO = 128, SBO = slab stride). Plus the small helpers these kernels share.
#pragma once
#include <cuda.h>
#include <cuda_fp16.h>

#include "common.cuh"
#include "tc_common.cuh"

namespace lawcat {
namespace ctc {

using namespace tc;

constexpr int TT = 128;   // tokens per tile
constexpr int HALO = 3;   // raw rows kept in front of a tile (conv width up to 4)
// |y| below which exp(y) is formed without the row's maximum (exp(24) is far from any limit; 16-bit features take 2^(y log2(e)), whose
// argument is rounded by up to 2^-19: 1.3e-6 of a feature, which is then rounded to bf16, 2e-3)
constexpr float Y_MAX = 24.f;

// Grid of the kernels that take one (sequence, head) and one tile of TT tokens per block: x the (sequence, head), whose number
// may pass the 65535 that end the other axes, y and z the tile.
inline dim3 tile_grid(int heads, int T) {
  const unsigned tiles = (unsigned)(T + TT - 1) / TT, y = tiles < 32768u ? tiles : 32768u;
  return dim3((unsigned)heads, y, (tiles + y - 1) / y);
}
__device__ __forceinline__ int tile_of_block() { return (int)(blockIdx.z * gridDim.y + blockIdx.y); }

template <int D>
struct Lay {
  static constexpr int OPR = D / 8;                         // 16-byte octets per row
  static constexpr uint32_t SLAB_W = D * 16 + 16;           // slab stride of the W tile (D rows)
  static constexpr uint32_t SLAB_U = TT * 16 + 16;          // slab stride of tiles with 128 token rows
  static constexpr uint32_t TILE_W = OPR * SLAB_W, TILE_U = OPR * SLAB_U;
  static constexpr uint32_t RAW_STRIDE = D * 2 + 16;        // bytes per raw row (padded: the conv reads 4 rows per warp)
  static constexpr uint32_t RAW_BYTES = (TT + HALO) * RAW_STRIDE;
};

__device__ __forceinline__ uint32_t toff(uint32_t slab, int r, int c) { return (uint32_t)(c >> 3) * slab + (uint32_t)r * 16u + (uint32_t)(c & 7) * 2u; }
__device__ __forceinline__ uint64_t kview(uint32_t addr, uint32_t slab) { return smem_desc(addr, slab, 128, LAYOUT_NONE); }
__device__ __forceinline__ uint64_t mview(uint32_t addr, uint32_t slab) { return smem_desc(addr, 128, slab, LAYOUT_NONE); }
__device__ __forceinline__ uint64_t dadv(uint64_t d, uint32_t bytes) {
  return (d & 0xFFFFFFFF00000000ull) | (uint64_t)((uint32_t)d + (bytes >> 4));
}
__device__ __forceinline__ void unpack8b(const uint4& v, float* f) {
  f[0] = bf16_lo(v.x); f[1] = bf16_hi(v.x); f[2] = bf16_lo(v.y); f[3] = bf16_hi(v.y);
  f[4] = bf16_lo(v.z); f[5] = bf16_hi(v.z); f[6] = bf16_lo(v.w); f[7] = bf16_hi(v.w);
}
__device__ __forceinline__ uint4 pack8f16(const float* v) {
  return make_uint4(pack_f16(v[0], v[1]), pack_f16(v[2], v[3]), pack_f16(v[4], v[5]), pack_f16(v[6], v[7]));
}
__device__ __forceinline__ uint4 pack8bf16(const float* v) {
  return make_uint4(pack_bf16(v[0], v[1]), pack_bf16(v[2], v[3]), pack_bf16(v[4], v[5]), pack_bf16(v[6], v[7]));
}
__device__ __forceinline__ void store_row8(bf16* p, const float* v) { *reinterpret_cast<uint4*>(p) = pack8bf16(v); }
__device__ __forceinline__ void store_row8(float* p, const float* v) {
  *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
  *reinterpret_cast<float4*>(p + 4) = make_float4(v[4], v[5], v[6], v[7]);
}
__device__ __forceinline__ void load_row8(const bf16* p, float* v) { unpack8b(*reinterpret_cast<const uint4*>(p), v); }
__device__ __forceinline__ void load_row8(const float* p, float* v) {
  const float4 a = *reinterpret_cast<const float4*>(p), b = *reinterpret_cast<const float4*>(p + 4);
  v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
}

// eight consecutive floats at a 32-byte boundary by one load: as two, each would take half of every sector it touches
__device__ __forceinline__ void load_octet(const float* p, float4 (&v)[2]) {
  asm volatile("ld.global.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=f"(v[0].x), "=f"(v[0].y), "=f"(v[0].z), "=f"(v[0].w), "=f"(v[1].x), "=f"(v[1].y), "=f"(v[1].z), "=f"(v[1].w)
               : "l"(p)
               : "memory");
}

__device__ __forceinline__ float log2_sigmoid(float a) {
  const float x = -a * 1.4426950408889634f;
  return -fmaxf(x, lg2f(1.f + ex2f(fminf(x, 126.f))));
}
__device__ __forceinline__ uint4 pack8h(const float* v, bool f16) {
  return f16 ? make_uint4(pack_f16(v[0], v[1]), pack_f16(v[2], v[3]), pack_f16(v[4], v[5]), pack_f16(v[6], v[7]))
             : make_uint4(pack_bf16(v[0], v[1]), pack_bf16(v[2], v[3]), pack_bf16(v[4], v[5]), pack_bf16(v[6], v[7]));
}
// 16-bit values back to fp32
__device__ __forceinline__ void unpack8h(const uint4& v, bool f16, float* f) {
  if (f16) {
    const __half2* h = reinterpret_cast<const __half2*>(&v);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float2 x = __half22float2(h[i]);
      f[2 * i] = x.x; f[2 * i + 1] = x.y;
    }
  } else {
    f[0] = bf16_lo(v.x); f[1] = bf16_hi(v.x); f[2] = bf16_lo(v.y); f[3] = bf16_hi(v.y);
    f[4] = bf16_lo(v.z); f[5] = bf16_hi(v.z); f[6] = bf16_lo(v.w); f[7] = bf16_hi(v.w);
  }
}
// v = hi + lo with hi the 16-bit rounding of v and lo the 16-bit rounding of the rest
__device__ __forceinline__ void split8h(const float* v, bool f16, uint4& hi, uint4& lo) {
  hi = pack8h(v, f16);
  float h[8], r[8];
  unpack8h(hi, f16, h);
#pragma unroll
  for (int i = 0; i < 8; ++i) r[i] = v[i] - h[i];
  lo = pack8h(r, f16);
}
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, float* v) {
  uint32_t r[8];
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr)
               : "memory");
#pragma unroll
  for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(r[i]);
}
__device__ __forceinline__ void tmem_st8(uint32_t taddr, const float* v) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
               ::"r"(taddr), "r"(__float_as_uint(v[0])), "r"(__float_as_uint(v[1])), "r"(__float_as_uint(v[2])),
                 "r"(__float_as_uint(v[3])), "r"(__float_as_uint(v[4])), "r"(__float_as_uint(v[5])),
                 "r"(__float_as_uint(v[6])), "r"(__float_as_uint(v[7]))
               : "memory");
}

// one mbarrier, bounded wait (a product batch completes within microseconds; 2e8 cycles is about a tenth of a second)
struct Waiter {
  uint32_t bar, phase;
  volatile int* abort_flag;
  int* dev_status;
  __device__ __forceinline__ void wait() {
    if (!*abort_flag) {
      bool ok = mbar_try_wait(bar, phase);
      if (!ok) {
        const long long t0 = clock64();
        while (!ok) {
#pragma unroll 1
          for (int i = 0; i < 16 && !ok; ++i) ok = mbar_try_wait(bar, phase);
          if (!ok && (*abort_flag || clock64() - t0 > 200000000LL)) break;
        }
      }
      if (!ok) {
        *abort_flag = 1;
        if (dev_status) atomicMax(dev_status, (int)LAWCAT_ERR_TIMEOUT);
      }
    }
    phase ^= 1u;
    tc_fence_after_sync();
  }
};

// W[h][c][e] (bf16, exact in fp16) as a tile with rows c, columns e
template <int D>
__device__ __forceinline__ void load_w_tile(uint8_t* s_wt, const bf16* Wh, int tid, int nthreads) {
  using L = Lay<D>;
  for (int idx = tid; idx < D * L::OPR; idx += nthreads) {
    const int c = idx / L::OPR, o = idx % L::OPR;
    float f[8];
    unpack8b(*reinterpret_cast<const uint4*>(Wh + (size_t)c * D + o * 8), f);
    *reinterpret_cast<uint4*>(s_wt + toff(L::SLAB_W, c, o * 8)) = pack8f16(f);
  }
}

// hint: fetch the 128-byte line at p towards L2 (these kernels walk their tiles in lock-step; the hint lets the next
// tile's rows travel while the current one is computed)
__device__ __forceinline__ void prefetch_l2(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }

// Conv of 8 channels (octet o) of N consecutive tokens from t on, straight from global memory: the window of raw rows (rows
// before the sequence come from the conv cache or are zero, rows past its end are zero), loaded well before its use ...
template <int D, int N>
__device__ __forceinline__ void conv_load(uint4 (&raw)[N + HALO], const bf16* x, const bf16* cache, int b, int t, int T, int NH,
                                          int head, int K, int o) {
#pragma unroll
  for (int i = 0; i < N + HALO; ++i) {
    const int tt = t - HALO + i;
    raw[i] = make_uint4(0u, 0u, 0u, 0u);
    if (tt >= 0 && tt < T)
      raw[i] = *reinterpret_cast<const uint4*>(x + (((size_t)b * T + tt) * NH + head) * D + o * 8);
    else if (tt < 0 && cache != nullptr && tt + (K - 1) >= 0)
      raw[i] = *reinterpret_cast<const uint4*>(cache + (((size_t)b * (K - 1) + tt + (K - 1)) * NH + head) * D + o * 8);
  }
}
// A head's taps as packed pairs of channels, fp32 (zero beyond the conv width): the pairs of taps (dl, dl + 1) of channel pair cp
// of octet o are the 16 bytes at ((2 cp + dl / 2) * D / 8 + o) * 16, so that neighbouring octets lie side by side. (As [D][4] rows
// the eight lanes of a quarter warp met in four banks: more than half of all shared-memory wavefronts of these kernels.)
template <int D>
__device__ __forceinline__ void load_taps(uint8_t* s_taps, const bf16* w, int head, int K, int tid, int nthreads) {
  for (int idx = tid; idx < D * 2; idx += nthreads) {
    const int o = idx % (D / 8), cp = idx / (D / 8) & 3, dl = idx / (D / 2);
    const bf16* wc = w + ((size_t)head * D + o * 8 + 2 * cp) * K + dl;
    const uint64_t t = dl < K ? f2_pack(__bfloat162float(wc[0]), __bfloat162float(wc[K])) : f2_pack(0.f, 0.f);
    *reinterpret_cast<uint64_t*>(s_taps + ((2 * cp + (dl >> 1)) * (D / 8) + o) * 16 + (dl & 1) * 8) = t;
  }
}
__device__ __forceinline__ void unpack8p(const uint4& v, uint64_t* f) {  // 8 bf16 values -> 4 packed pairs of fp32
  f[0] = f2_pack(bf16_lo(v.x), bf16_hi(v.x)); f[1] = f2_pack(bf16_lo(v.y), bf16_hi(v.y));
  f[2] = f2_pack(bf16_lo(v.z), bf16_hi(v.z)); f[3] = f2_pack(bf16_lo(v.w), bf16_hi(v.w));
}
// ... and the sums, in pairs of channels; emit(i, u) takes token t + i. Every raw row is unpacked once.
template <int D, int N, typename F>
__device__ __forceinline__ void conv_emit(const uint4 (&raw)[N + HALO], const uint8_t* s_taps, int o, F emit) {
  uint64_t w[4][4], x0[4], x1[4], x2[4], x3[4];
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    const ulonglong2 t = *reinterpret_cast<const ulonglong2*>(s_taps + (u * (D / 8) + o) * 16);
    w[u >> 1][2 * (u & 1)] = t.x;
    w[u >> 1][2 * (u & 1) + 1] = t.y;
  }
  unpack8p(raw[0], x3); unpack8p(raw[1], x2); unpack8p(raw[2], x1);
#pragma unroll
  for (int i = 0; i < N; ++i) {
    uint64_t u[4];
    unpack8p(raw[i + HALO], x0);
#pragma unroll
    for (int cp = 0; cp < 4; ++cp)
      u[cp] = f2_fma(w[cp][3], x3[cp], f2_fma(w[cp][2], x2[cp], f2_fma(w[cp][1], x1[cp], f2_mul(w[cp][0], x0[cp]))));
    emit(i, u);
#pragma unroll
    for (int cp = 0; cp < 4; ++cp) { x3[cp] = x2[cp]; x2[cp] = x1[cp]; x1[cp] = x0[cp]; }
  }
}
__device__ __forceinline__ void pairs_to_floats(const uint64_t* v, float* f) {
#pragma unroll
  for (int i = 0; i < 4; ++i) f2_unpack(v[i], f[2 * i], f[2 * i + 1]);
}

// v rounded to bf16, and v -= the rounded value
__device__ __forceinline__ uint4 take_bf16(uint64_t* v) {
  float f[8];
  uint64_t h[4];
  pairs_to_floats(v, f);
  const uint4 p = pack8bf16(f);
  unpack8p(p, h);
  const uint64_t neg = f2_pack(-1.f, -1.f);
#pragma unroll
  for (int i = 0; i < 4; ++i) v[i] = f2_fma(h[i], neg, v[i]);
  return p;
}

}  // namespace ctc
}  // namespace lawcat
