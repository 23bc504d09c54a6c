// Linear-attention context module.
//
// The online deployment of the paper (Appendix B.3) serves 1,000-interaction
// contexts with linear attention (Katharopoulos et al., 2020).  Here it
// replaces the softmax in the element -> context cross-attention of Section
// 4.2: with the feature map phi(x) = elu(x) + 1, non-causal over the
// context, the context of a request reduces, per layer l and head h, to the
// state
//     S = sum_c phi(K_l[c, h]) V_l[c, h]^T   [d_h, d_h],   z = sum_c phi(K_l[c, h])   [d_h],
// computed once per request (the QKV-Cache idea with a constant-size state
// instead of C key/value rows), and an element query q reads
//     a = phi(q) S / (phi(q) . z).
//
//   lin_state_kernel : one CTA per (segment, layer, group of up to 128
//                      features); streams the segment's C key/value rows
//                      through operand tiles of 64 rows, phi(K)^T [V | 1] on
//                      the tensor core
//   lin_attn_kernel  : one to eight CTAs per segment; the segment's states of
//                      one layer (all heads) and phi(q) of 16- to 64-row
//                      blocks in shared memory, one warp per (head, 8 rows), a
//                      lane per output column and 8 rows of accumulators in
//                      registers
#include <cuda_fp16.h>

#include "fe_common.cuh"
#include "fe_kernels.h"

namespace fe {

namespace {

__device__ __forceinline__ float pow2(int n) { return __int_as_float((127 + n) << 23); }  // |n| <= 126

// f16 value as an integer of the same order
__device__ __forceinline__ int order_key(__half x) {
  const int b = __half_as_short(x);
  return b >= 0 ? b : b ^ 0x7FFF;
}
__device__ __forceinline__ __half order_half(int k) { return __short_as_half((short)(k >= 0 ? k : k ^ 0x7FFF)); }

// elu(x) + 1; the exponential branch (x <= 0, result in (0, 1]) through the
// hardware exponent unit, whose relative error is far below the f16 rounding
// of the keys and queries it is applied to
__device__ __forceinline__ float phi(float x) { return x > 0.f ? x + 1.f : __expf(x); }

constexpr int kChunk = 64;                // context rows per operand tile
constexpr uint32_t kAtom = kChunk * 128;  // 64 features x kChunk rows, f16
constexpr int kFlush = 16;                // chunks that are added up on the tensor core (even)
constexpr float kLoScale = 2048.f;        // phi's lo plane is stored times 2^11 (at most 2^15)
constexpr float kPhiSmall = 1.f / 8192;   // 2^-13
constexpr float kKeySmall = -9.f;         // keys below: phi < 2^-12.98

// MN-major operand descriptor, 128-byte swizzle: atoms of 64 features, kAtom apart, 8-row groups 1024 bytes apart
__device__ __forceinline__ uint64_t desc_feat(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);
  d |= (uint64_t)(kAtom >> 4) << 16;
  d |= (uint64_t)(1024 >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)2 << 61;
  return d;
}

// operand tiles of a chunk: phi(K) hi and lo (128 features each), V and the ones columns
template <int FG>
struct StateCfg {
  static constexpr uint32_t kA = 2 * kAtom;
  static constexpr uint32_t kV = (FG == 128 ? 3 : FG == 64 ? 2 : 1) * kAtom;
  static constexpr uint32_t kBuf = 2 * kA + kV;
  static constexpr size_t kSmem = 2 * kBuf + 64 + FG * 4;  // two buffers, barriers, each feature's largest key
  // three accumulators: the hi products of even and of odd chunks, the lo products;
  // 512 columns for FG = 128 (one CTA on an SM at a time), 256 below
  static constexpr int kN = FG + 16;
  static constexpr uint32_t kCols = 3 * kN <= 256 ? 256 : 512;
};

}  // namespace

// Context states.  A CTA takes one segment, one layer and one group of FG
// features (FG = min(d, 128): the heads [g FG / DH, (g + 1) FG / DH)).  Per
// 64 context rows its threads write phi(K), as a hi + lo pair of f16 tiles, and V,
// an exact f16 tile followed by 16 columns of ones, and the tensor core adds
// phi(K)^T [V | 1] to 128 x (FG + 16) accumulators in TMEM (z comes from the ones
// columns).  Two operand buffers: the next chunk's rows are transformed and
// written while the current one is multiplied, and the rows of two chunks are in flight.
//
// Precision: hi + lo hold 22 bits of phi for phi >= 2^-14 (lo is stored times 2^11
// and its accumulator scaled back), and below that all but 2^-36.  A feature whose
// largest phi over the context is below 2^-13 would lose bits, and below 2^-36 all of
// them, so such a segment's group (z / C tells) is done over with each of those
// features' phi times a power of two that brings its largest one to (1/2, 1], undone
// in the stored state.  The tensor core truncates each addition to its accumulator, so there are three
// (hi of even and of odd chunks, lo), and their sums go to the stored state, added in
// fp32, every 16 chunks.  Relative error of S (2-norm) and largest of z against 64 bits, 1000
// rows: 6.2e-7, 1e-7 with keys ~ N(0, 0.5), 6.3e-7, 2e-7 at mean -12, 6.2e-7, 3e-7 at -20,
// 8.7e-7, 6e-7 at -40; a chain of fp32 multiply-adds per element: 5.7e-7, 1.1e-6;
// 6.4e-7, 1.8e-6; 7.3e-7, 1.9e-6; 1.1e-6, 1.5e-6.
// 2000 rows: 6.2e-7 (7.7e-7).
//
// What bounds it: the transform of K (an exponent, two conversions and a 16-byte
// store per plane for 8 values); the products take 8 MMAs of N = FG + 16 a chunk.
// 256 segments of 1000 rows, two layers of 64 columns: 107 us with fp32 products on the
// CUDA cores, 57 here (131 MB of K/V, 20 us at the copy rate; 54 without the scaled lo
// plane, the test of z and the flushes), the 512 CTAs being 1.7 waves of two per SM.
// FG = 128: 181 -> 151 at d = 128; there a CTA takes all of the SM's TMEM columns (3 x 144 of
// 512), so a second one on the SM waits for the first to end.
template <int DH, int FG>
__global__ void __launch_bounds__(256, 2) lin_state_kernel(const __half* __restrict__ kv, int hm, int rows_alloc,
                                                           int ld, int C, int d, int H, float* __restrict__ states,
                                                           int* status) {
  using Cfg = StateCfg<FG>;
  constexpr int HG = FG / DH;               // heads per group
  constexpr int SB = DH * DH + DH;
  constexpr int NP = kChunk * FG / 8;       // 16-byte pieces of a chunk, for K and for V
  constexpr int P8 = NP / 256;              // per thread
  static_assert(NP % 256 == 0, "tiling");
  extern __shared__ __align__(1024) uint8_t sm_state[];
  uint64_t* bars = reinterpret_cast<uint64_t*>(sm_state + 2 * Cfg::kBuf);
  uint64_t* free_bar = bars;                // [2] the products of the chunk in this buffer are complete
  uint64_t* drain = bars + 2;               // the products in flight at the end
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 3);
  int* kmax = reinterpret_cast<int*>(bars + 8);  // [FG] each feature's largest key of the segment (order_key)
  const int s = blockIdx.x, G = d / FG, l = blockIdx.y / G, g = blockIdx.y % G;
  const int kcol = 2 * l * d + g * FG, vcol = (2 * l + 1) * d + g * FG;
  const size_t row0 = (size_t)s * C;
  // element (row, col) of K/V: head-major blocks [col / DH][rows_alloc][DH], or row-major [rows][ld]
  auto at = [&](size_t row, int col) -> size_t {
    return hm ? ((size_t)(col / DH) * rows_alloc + row) * DH + (col % DH) : row * ld + col;
  };
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  // the 16-byte piece of (row r, features m .. m + 7) in an operand tile
  auto piece = [](int r, int m) {
    return (uint32_t)(m >> 6) * kAtom + (uint32_t)r * 128u + ((((uint32_t)(m & 63) >> 3) ^ (uint32_t)(r & 7)) << 4);
  };
  if (t == 0) {
    mbar_init(free_bar, 1);
    mbar_init(free_bar + 1, 1);
    mbar_init(drain, 1);
    fence_mbar_init();
  }
  if (t < FG) kmax[t] = order_key(__ushort_as_half(0xFC00u));  // -inf
  if (warp == 0) tmem_alloc(tmem_slot, Cfg::kCols);
  // features FG .. 127 of phi(K) are zeros, V's columns FG .. FG + 15 ones
  for (int i = t; i < 2 * kChunk; i += 256) {
    const int r = i % kChunk;
    uint8_t* buf = sm_state + (size_t)(i / kChunk) * Cfg::kBuf;
    for (int m = FG; m < 128; m += 8) {
      *reinterpret_cast<uint4*>(buf + piece(r, m)) = make_uint4(0u, 0u, 0u, 0u);
      *reinterpret_cast<uint4*>(buf + Cfg::kA + piece(r, m)) = make_uint4(0u, 0u, 0u, 0u);
    }
    const uint32_t one2 = 0x3C003C00u;
    *reinterpret_cast<uint4*>(buf + 2 * Cfg::kA + piece(r, FG)) = make_uint4(one2, one2, one2, one2);
    *reinterpret_cast<uint4*>(buf + 2 * Cfg::kA + piece(r, FG + 8)) = make_uint4(one2, one2, one2, one2);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  // the 16-byte pieces of a chunk this thread loads; rows past C read as zero
  auto load = [&](int r0, uint4* kr, uint4* vr) {
#pragma unroll
    for (int q = 0; q < P8; ++q) {
      const int idx = t + 256 * q, r = idx / (FG / 8), c8 = (idx % (FG / 8)) * 8;
      if (r0 + r < C) {
        kr[q] = *reinterpret_cast<const uint4*>(kv + at(row0 + r0 + r, kcol + c8));
        vr[q] = *reinterpret_cast<const uint4*>(kv + at(row0 + r0 + r, vcol + c8));
      } else {
        kr[q] = make_uint4(0u, 0u, 0u, 0u);
        vr[q] = kr[q];
      }
    }
  };
  const uint32_t go = elect_one();
  const uint32_t idesc = umma_idesc_f16(128, Cfg::kN) | (1u << 15) | (1u << 16);  // A and B MN-major
  float scale[8];  // of this thread's features' phi, in a second pass
  int used[2] = {0, 0};  // chunks put through each operand buffer
  // chunk it (its pieces in kr, vr; chunk it + 2's are then loaded into them) through operand buffer B
  auto chunk = [&](auto bufc, auto scaled, int it, uint4* kr, uint4* vr) {
    constexpr int B = decltype(bufc)::value;
    constexpr bool kScaled = decltype(scaled)::value;
    const int r0 = it * kChunk;
    uint8_t* buf = sm_state + (size_t)B * Cfg::kBuf;
    if (used[B] > 0) mbar_wait_role(free_bar + B, (uint32_t)(used[B] - 1) & 1u, status);
    ++used[B];
#pragma unroll
    for (int q = 0; q < P8; ++q) {
      const int idx = t + 256 * q, r = idx / (FG / 8), c8 = (idx % (FG / 8)) * 8;
      const bool valid = r0 + r < C;  // a missing row adds nothing
      const __half2* hk = reinterpret_cast<const __half2*>(&kr[q]);
      uint32_t hi[4], lo[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const float2 x = __half22float2(hk[e]);
        float f0 = valid ? phi(x.x) : 0.f, f1 = valid ? phi(x.y) : 0.f;
        if (kScaled) {
          f0 *= scale[2 * e];
          f1 *= scale[2 * e + 1];
        }
        const __half2 h = __floats2half2_rn(f0, f1);
        const float2 hf = __half22float2(h);
        hi[e] = *reinterpret_cast<const uint32_t*>(&h);
        lo[e] = pack_f16x2((f0 - hf.x) * kLoScale, (f1 - hf.y) * kLoScale);
      }
      *reinterpret_cast<uint4*>(buf + piece(r, c8)) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
      *reinterpret_cast<uint4*>(buf + Cfg::kA + piece(r, c8)) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
      *reinterpret_cast<uint4*>(buf + 2 * Cfg::kA + piece(r, c8)) = vr[q];
    }
    fence_async_shared();
    tc_fence_before();
    __syncthreads();
    if (r0 + 2 * kChunk < C) load(r0 + 2 * kChunk, kr, vr);  // in flight for a whole chunk (issued before the fence, it waited for them)
    if (warp == 0) {
      tc_fence_after();
      const uint64_t ah = desc_feat(smem_u32(buf)), al = desc_feat(smem_u32(buf + Cfg::kA)),
                     bd = desc_feat(smem_u32(buf + 2 * Cfg::kA));
#pragma unroll
      for (int kk = 0; kk < kChunk / 16; ++kk) {
        const uint32_t o = (uint32_t)kk * 16u * 128u;
        umma_bf16_if(tmem + (uint32_t)(B * Cfg::kN), desc_adv(ah, o), desc_adv(bd, o), idesc,
                     (it % kFlush > 1 || kk != 0) ? 1u : 0u, go);
        umma_bf16_if(tmem + 2u * Cfg::kN, desc_adv(al, o), desc_adv(bd, o), idesc, (it % kFlush | kk) != 0 ? 1u : 0u, go);
      }
      umma_commit_if(free_bar + B, go);
    }
  };
  // The sums of the chunks since the last flush (up to number `last`) to the stored state, added to
  // what it holds unless they are the first.  Lane m of the accumulators: feature m of the
  // group; its head's DH columns, and z in column FG.
  const int q = warp & 3, sub = warp >> 2, m = 32 * q + lane;
  const int Ly = gridDim.y / G;
  // S row-major, then z
  float* st = states + (((size_t)s * Ly + l) * H + g * HG + (m < FG ? m / DH : 0)) * SB;
  const bool z_warp = 32 * q < FG && sub == (DH == 64 ? 0 : 1);  // holds z of feature m
  // every product up to chunk `last`'s complete
  auto settle = [&](int last) {
    const int lb = last & 1;
    mbar_wait_role(free_bar + lb, (uint32_t)((lb ? used[1] : used[0]) - 1) & 1u, status);
    tc_fence_after();
  };
  // z of feature m up to chunk `last` (a z_warp's)
  auto z_sum = [&](int last) {
    const uint32_t row = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)FG;
    uint32_t z[8], w[8], u[8];
    tmem_ld8(row, z);
    tmem_ld8(row + (uint32_t)Cfg::kN, u);
    tmem_ld8(row + (uint32_t)(2 * Cfg::kN), w);
    float x = fmaf(__uint_as_float(w[0]), 1.f / kLoScale, __uint_as_float(z[0]));
    if (last % kFlush > 0) x += __uint_as_float(u[0]);
    return last >= kFlush ? st[DH * DH + m % DH] + x : x;
  };
  auto flush = [&](int last, float f) {
    settle(last);
    const bool add = last >= kFlush;
    const bool odd = last % kFlush > 0;  // (a single chunk leaves the second accumulator unwritten)
    if (32 * q < FG) {
      const int i = m % DH;
      const uint32_t row = tmem + ((uint32_t)(q * 32) << 16);
      if (sub == 0 || DH == 64) {
#pragma unroll 1
        for (int c = 0; c < 32; c += 8) {
          const uint32_t col = row + (uint32_t)((32 * q) / DH * DH + 32 * sub + c);
          float* dst = st + i * DH + 32 * sub + c;
          uint32_t v[8], w[8];
          float x[8];
          tmem_ld8(col, v);
          tmem_ld8(col + 2u * Cfg::kN, w);
#pragma unroll
          for (int j = 0; j < 8; ++j) x[j] = fmaf(__uint_as_float(w[j]), 1.f / kLoScale, __uint_as_float(v[j]));
          if (odd) {
            tmem_ld8(col + (uint32_t)Cfg::kN, w);
#pragma unroll
            for (int j = 0; j < 8; ++j) x[j] += __uint_as_float(w[j]);
          }
          if (add) {
#pragma unroll
            for (int j = 0; j < 8; ++j) x[j] += dst[j];
          }
#pragma unroll
          for (int j = 0; j < 8; j += 4)
            *reinterpret_cast<float4*>(dst + j) = make_float4(x[j] * f, x[j + 1] * f, x[j + 2] * f, x[j + 3] * f);
        }
      }
    }
    if (z_warp) st[DH * DH + m % DH] = z_sum(last) * f;
    tc_fence_before();
    __syncthreads();  // the accumulators are read
  };
  uint4 k0[P8], v0[P8], k1[P8], v1[P8];
  const int it_end = (C + kChunk - 1) / kChunk;
  // every chunk; the last window's sums stay in the accumulators
  auto pass = [&](auto scaled) {
    load(0, k0, v0);
    load(kChunk, k1, v1);
    for (int i = 0; i < it_end; i += 2) {
      if (i > 0 && i % kFlush == 0) flush(i - 1, 1.f);
      chunk(std::integral_constant<int, 0>{}, scaled, i, k0, v0);
      if (i + 1 < it_end) chunk(std::integral_constant<int, 1>{}, scaled, i + 1, k1, v1);
    }
  };
  pdl_trigger();
  pdl_wait();
  pass(std::false_type{});
  // A feature with z >= 2^-13 C has a phi of 2^-13 or more.  Where one has not: each feature's
  // largest key, and with it the power of two of its phi (1 if that is 2^-13 or more)
  float f = 1.f;
  settle(it_end - 1);
  const bool low = z_warp && z_sum(it_end - 1) < kPhiSmall * (float)C;
  tc_fence_before();
  if (__syncthreads_or(low)) {
    __half2 km[4];  // of this thread's 8 features
#pragma unroll
    for (int e = 0; e < 4; ++e) km[e] = __half2half2(__ushort_as_half(0xFC00u));
    for (int i = t; i < C * (FG / 8); i += 256) {
      const uint4 k = *reinterpret_cast<const uint4*>(kv + at(row0 + i / (FG / 8), kcol + (i % (FG / 8)) * 8));
      const __half2* hk = reinterpret_cast<const __half2*>(&k);
#pragma unroll
      for (int e = 0; e < 4; ++e) km[e] = __hmax2(km[e], hk[e]);
    }
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      atomicMax(kmax + (t % (FG / 8)) * 8 + 2 * e, order_key(__low2half(km[e])));
      atomicMax(kmax + (t % (FG / 8)) * 8 + 2 * e + 1, order_key(__high2half(km[e])));
    }
    __syncthreads();
    auto exponent = [&](int mm) {
      const float x = __half2float(order_half(kmax[mm]));
      return x >= kKeySmall ? 0 : (int)fminf(126.f, floorf(-x * 1.44269504f));
    };
    if (__syncthreads_or(t < FG && exponent(t) != 0)) {
#pragma unroll
      for (int e = 0; e < 8; ++e) scale[e] = pow2(exponent((t % (FG / 8)) * 8 + e));
      pass(std::true_type{});
      if (m < FG) f = pow2(-exponent(m));
    }
  }
  flush(it_end - 1, f);
  if (warp == 0) {
    umma_drain(drain, status, go);
    tmem_dealloc(tmem, Cfg::kCols);
  }
}

namespace {
constexpr int kRowBlock = 64;  // element rows staged per block of lin_attn_kernel, at most
constexpr int kRowTask = 8;    // rows per warp task (a task: one head, kRowTask rows)
}

template <int DH>
__global__ void __launch_bounds__(256) lin_attn_kernel(const __half* __restrict__ q, int ldq, int d,
                                                       const float* __restrict__ states, int Ly, int l, int H,
                                                       const int* __restrict__ off_dev, const int* __restrict__ cnt_dev,
                                                       int stride, int cnt_fixed, int row_block, bf16* o_h, bf16* o_l,
                                                       int ldo) {
  constexpr int SB = DH * DH + DH;
  constexpr int NJ = DH / 32;           // output columns per lane
  extern __shared__ __align__(16) float sm[];
  float* sst = sm;                      // [H][SB]: layer l's states of this segment
  float* sq = sm + H * SB;              // [row_block][d + 4]: phi(q) of a block of rows (padded rows)
  const int ldq_s = d + 4;
  const int s = blockIdx.x;
  pdl_wait();
  pdl_trigger();
  const int off = off_dev ? off_dev[s] : s * stride;
  const int cnt = cnt_dev ? cnt_dev[s] : cnt_fixed;
  if ((int)blockIdx.y * row_block >= cnt) return;
  // the states, four 16-byte loads in flight per thread at a time
  {
    const float4* src = reinterpret_cast<const float4*>(states + ((size_t)s * Ly + l) * H * SB);
    float4* dst = reinterpret_cast<float4*>(sst);
    const int n4 = H * SB / 4;
    for (int i0 = threadIdx.x; i0 < n4; i0 += 1024) {
      float4 v[4];
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (i0 + 256 * u < n4) v[u] = src[i0 + 256 * u];
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (i0 + 256 * u < n4) dst[i0 + 256 * u] = v[u];
    }
  }
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int d8 = d / 8;
  for (int rb = blockIdx.y * row_block; rb < cnt; rb += gridDim.y * row_block) {
    const int nr = min(row_block, cnt - rb);
    __syncthreads();  // the previous block (and, the first time, the states) consumed / written
    for (int i0 = threadIdx.x; i0 < nr * d8; i0 += 1024) {
      uint4 raw[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int idx = i0 + 256 * u;
        if (idx < nr * d8) raw[u] = *reinterpret_cast<const uint4*>(q + (size_t)(off + rb + idx / d8) * ldq + (idx % d8) * 8);
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int idx = i0 + 256 * u;
        if (idx < nr * d8) {
          const int r = idx / d8, c8 = (idx % d8) * 8;
          const __half* hq = reinterpret_cast<const __half*>(&raw[u]);
#pragma unroll
          for (int e = 0; e < 8; ++e) sq[r * ldq_s + c8 + e] = phi(__half2float(hq[e]));
        }
      }
    }
    __syncthreads();
    // warp tasks (head, kRowTask rows of the block): lane j owns output
    // column j (and j + 32) of every row of its task
    const int nsub = (nr + kRowTask - 1) / kRowTask;
    for (int task = warp; task < H * nsub; task += 8) {
      const int h = task % H, sr = (task / H) * kRowTask;
      const float* S = sst + h * SB;
      const float* z = S + DH * DH;
      const float* qh = sq + sr * ldq_s + h * DH;
      const int tn = min(kRowTask, nr - sr);
      float acc[kRowTask][NJ];
#pragma unroll
      for (int r = 0; r < kRowTask; ++r)
#pragma unroll
        for (int jj = 0; jj < NJ; ++jj) acc[r][jj] = 0.f;
#pragma unroll 1
      for (int i = 0; i < DH; i += 4) {
        float sv[4][NJ];
#pragma unroll
        for (int ii = 0; ii < 4; ++ii)
#pragma unroll
          for (int jj = 0; jj < NJ; ++jj) sv[ii][jj] = S[(i + ii) * DH + lane + 32 * jj];
#pragma unroll
        for (int r = 0; r < kRowTask; ++r) {
          const float4 f = *reinterpret_cast<const float4*>(qh + r * ldq_s + i);  // one address: broadcast
#pragma unroll
          for (int jj = 0; jj < NJ; ++jj) {
            acc[r][jj] = fmaf(f.x, sv[0][jj], acc[r][jj]);
            acc[r][jj] = fmaf(f.y, sv[1][jj], acc[r][jj]);
            acc[r][jj] = fmaf(f.z, sv[2][jj], acc[r][jj]);
            acc[r][jj] = fmaf(f.w, sv[3][jj], acc[r][jj]);
          }
        }
      }
      // lane r: the normaliser phi(q_r) . z of row r (padded rows: conflict-free)
      float den = 0.f;
      if (lane < tn) {
#pragma unroll 4
        for (int i = 0; i < DH; i += 4) {
          const float4 f = *reinterpret_cast<const float4*>(qh + lane * ldq_s + i);
          den = fmaf(f.x, z[i], den);
          den = fmaf(f.y, z[i + 1], den);
          den = fmaf(f.z, z[i + 2], den);
          den = fmaf(f.w, z[i + 3], den);
        }
      }
#pragma unroll
      for (int r = 0; r < kRowTask; ++r) {
        const float inv = 1.f / __shfl_sync(0xFFFFFFFFu, den, r);
        if (r < tn) {
          const size_t row = (size_t)(off + rb + sr + r);
#pragma unroll
          for (int jj = 0; jj < NJ; ++jj) {
            const float x = acc[r][jj] * inv;
            const __nv_bfloat16 hi = __float2bfloat16_rn(x);
            const __nv_bfloat16 lo = __float2bfloat16_rn(x - __bfloat162float(hi));
            const size_t o = row * ldo + h * DH + lane + 32 * jj;
            o_h[o] = hi;
            o_l[o] = lo;
          }
        }
      }
    }
  }
}

namespace {
// H <= 8 heads of d_h = 64, and a block of rows of width d <= 512 (half a block there)
int g_lin_sms = 0;
constexpr int kLinAttnSmemMax = 8 * (64 * 64 + 64) * 4 + kRowBlock / 2 * (512 + 4) * 4;
}

cudaError_t linattn_prepare() {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&g_lin_sms, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(lin_attn_kernel<32>, cudaFuncAttributeMaxDynamicSharedMemorySize, kLinAttnSmemMax);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(lin_attn_kernel<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, kLinAttnSmemMax);
  auto state = [&](const void* f, size_t smem) {
    if (e == cudaSuccess) e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  };
  state((const void*)lin_state_kernel<32, 128>, StateCfg<128>::kSmem);
  state((const void*)lin_state_kernel<32, 64>, StateCfg<64>::kSmem);
  state((const void*)lin_state_kernel<64, 128>, StateCfg<128>::kSmem);
  state((const void*)lin_state_kernel<64, 64>, StateCfg<64>::kSmem);
  state((const void*)lin_state_kernel<32, 32>, StateCfg<32>::kSmem);
  return e;
}

cudaError_t lin_state_launch(const bf16* kv, int hm, int rows_alloc, int ld, int n_seg, int C, int d, int dh, int Ly,
                             int H, float* states, int* status, cudaStream_t s) {
  if (n_seg <= 0 || C <= 0) return cudaSuccess;
  const int FG = d < 128 ? d : 128;
  const dim3 grid((unsigned)n_seg, (unsigned)(Ly * (d / FG)));
  const __half* k = reinterpret_cast<const __half*>(kv);
  auto go = [&](auto kern, size_t smem) {
    return launch_k(kern, grid, dim3(256), smem, s, k, hm, rows_alloc, ld, C, d, H, states, status);
  };
  if (dh == 32 && FG == 128) return go(lin_state_kernel<32, 128>, StateCfg<128>::kSmem);
  if (dh == 32 && FG == 64) return go(lin_state_kernel<32, 64>, StateCfg<64>::kSmem);
  if (dh == 64 && FG == 128) return go(lin_state_kernel<64, 128>, StateCfg<128>::kSmem);
  if (dh == 64 && FG == 64) return go(lin_state_kernel<64, 64>, StateCfg<64>::kSmem);
  if (dh == 32 && FG == 32) return go(lin_state_kernel<32, 32>, StateCfg<32>::kSmem);
  return cudaErrorInvalidValue;
}

cudaError_t lin_attn_launch(const bf16* q, int ldq, const float* states, int n_seg, int Ly, int l, int H, int dh,
                            const int* off_dev, const int* cnt_dev, int stride, int cnt_fixed, bf16* o_h, bf16* o_l,
                            int ldo, cudaStream_t s) {
  if (n_seg <= 0) return cudaSuccess;
  const int d = H * dh;
  // A CTA is a chain of two loads and a product per block of rows, so a segment's rows are dealt out to CTAs
  // until there are about four per SM (in all for 256 segments of 60 rows, d = 64: one CTA each and blocks of 32
  // rows, 16 per task, 190 us, blocks of 64 and 8 per task 186.4, two CTAs 178.1, more 178.0; for 64 segments
  // 120.1, 113.2, 109.3 with eight), in smaller blocks the more of them there are (64 segments of 100 rows, d =
  // 128: blocks of 32 190, of 16 185; 256 of 60, d = 64, with four CTAs: 178.0 and 180.5).
  int ny = 4 * (g_lin_sms > 0 ? g_lin_sms : 148) / n_seg;
  ny = ny < 1 ? 1 : ny > 8 ? 8 : ny;
  const int row_block = ny >= 4 ? kRowBlock / 4 : ny > 1 || d > 256 ? kRowBlock / 2 : kRowBlock;
  const size_t smem = ((size_t)H * (dh * dh + dh) + (size_t)row_block * (d + 4)) * sizeof(float);
  if (smem > (size_t)kLinAttnSmemMax) return cudaErrorInvalidValue;
  const __half* qh = reinterpret_cast<const __half*>(q);
  const dim3 grid((unsigned)n_seg, (unsigned)ny);
  if (dh == 32)
    return launch_k(lin_attn_kernel<32>, grid, dim3(256), smem, s, qh, ldq, d, states, Ly, l, H, off_dev, cnt_dev, stride,
                    cnt_fixed, row_block, o_h, o_l, ldo);
  if (dh == 64)
    return launch_k(lin_attn_kernel<64>, grid, dim3(256), smem, s, qh, ldq, d, states, Ly, l, H, off_dev, cnt_dev, stride,
                    cnt_fixed, row_block, o_h, o_l, ldo);
  return cudaErrorInvalidValue;
}

}  // namespace fe
