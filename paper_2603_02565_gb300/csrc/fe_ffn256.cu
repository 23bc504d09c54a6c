// Attention output projection and position-wise FFN of one block (the element
// layers of Section 4.2, the SeqEnc block of Section 4.3) for rows of width
// d = 256, in one kernel:
//     x = x0 + A W_O,   x_out = x + ReLU(LN(x) W1 + b1) W2 + b2,   LN(x_out),
// and optionally the next layer's query projection LN(x_out) W_Q (f16 out).
// x, LN(x) and the F-wide hidden activation never reach memory.
//
// At d = 256 the split LN(x) operand of a 128-row tile alone is 128 KB of
// shared memory, so every weight streams through a ring of five 16 KB boxes
// (128 rows x 64 columns, 128-byte swizzle) in the order the MMAs consume
// them, and every product is a sequence of N = 128 MMAs of one box each:
//   W_O  : k block kb, output half nh                       (8 boxes)
//   FFN1 : chunk f of 128 hidden units, k block kb          (4 boxes)
//   FFN2 : chunk f, output half nh, 64-unit half of the chunk (4 boxes)
//   W_Q  : as W_O (the tail)                                  (8 boxes)
// TMEM: columns [0, 256) take A W_O, then the two FFN1 chunk buffers
// (128 columns each), then the tail product; the d-column accumulator of x
// and FFN2 sits at [256, 512).  FFN1 of chunk f runs one chunk ahead of FFN2
// of chunk f - 1, which reads its A operand (the split ReLU output) from TMEM.
// Roles: warp 0 loads (TMA), warp 1 issues tcgen05.mma, warps
// 2-9 (two per TMEM lane quadrant, each owning 128 of a row's 256 columns)
// run the epilogues: x0 + projection, LayerNorm statistics exchanged with the
// partner warp, LN(x) as the split operand tile over the A tile, bias + ReLU
// + split per chunk, x_out + b2 (staged over the A tile and stored by TMA),
// LN(x_out) over the A tile (stored by TMA), and the tail's f16 output (over
// the upper half of the A tile, stored by TMA).  A tile's A and x0 are prefetched
// into L2 during the chunks of the tile before it, and each k block of the A tile
// is loaded as soon as the store that last used its memory has read it, so that
// A W_O starts while the rest is still on its way out or in.  Products take split
// bf16 activations (hi + lo) times exact bf16 weights with fp32 accumulation;
// LayerNorm and residuals are fp32.
// What bounds it: the tensor pipe (a chunk is 64 MMAs of N = 128, 4096 cycles, on
// both halves of its weights) and, per tile, the two LayerNorm phases.  A tile's first
// k block came 8.5k cycles after the previous tile's end (its stores drain at
// 32 bytes a cycle, then DRAM, on every SM at once), hence the prefetch and the
// release by k blocks; the epilogue loops stay rolled (127 registers, none spilled).
// 295k rows, a launch with the tail: 826 -> 566 us (tensor pipe 39 -> 55 %).
// Holding a thread's 128 columns in registers through both LayerNorm passes, the
// loops unrolled, was slower.
#include "fe_common.cuh"
#include "fe_kernels.h"

namespace fe {

namespace {
// TMA 2D load (predicated on go) with an L2 cache policy (createpolicy): evict_last for the weight
// boxes that every SM re-reads, evict_first for the activation tiles that
// stream past them once.
__device__ __forceinline__ void tma_load_2d_hint_if(void* smem_dst, const CUtensorMap* map, int x, int y,
                                                 uint64_t* bar, uint64_t policy, uint32_t go) {
  asm volatile(
      "{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %6, 0;\n\t"
      "@q cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint"
      " [%0], [%1, {%3, %4}], [%2], %5;\n\t}" ::"r"(smem_u32(smem_dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(smem_u32(bar)), "r"(x), "r"(y), "l"(policy), "r"(go)
      : "memory");
}
// all but the newest of this thread's bulk stores have read their source
__device__ __forceinline__ void bulk_wait_read1() { asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory"); }
// TMA 2D box into L2 only (predicated on go)
__device__ __forceinline__ void tma_prefetch_2d_if(const CUtensorMap* map, int x, int y, uint32_t go) {
  asm volatile(
      "{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %3, 0;\n\t"
      "@q cp.async.bulk.prefetch.tensor.2d.L2.global [%0, {%1, %2}];\n\t}" ::"l"(reinterpret_cast<uint64_t>(map)),
      "r"(x), "r"(y), "r"(go)
      : "memory");
}
__device__ __forceinline__ uint64_t l2_policy_evict_last() {
  uint64_t p;
  asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
  return p;
}
__device__ __forceinline__ uint64_t l2_policy_evict_first() {
  uint64_t p;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
  return p;
}

constexpr int BM = 128;
constexpr int BK = 64;
constexpr int D = 256;
constexpr int NKB = D / BK;   // 4
constexpr int FC = 128;       // hidden units per chunk
constexpr int kEpiWarps = 8;
constexpr int kThreads = 64 + 32 * kEpiWarps;  // 320
constexpr uint32_t kBox = BM * BK * 2;         // 16 KB
constexpr uint32_t kABytes = NKB * 2 * kBox;   // 128 KB: the split tile [kb][plane]
constexpr int kMaxF = 2048;
constexpr int kRing = 5;
constexpr uint32_t kOffMisc = kABytes + kRing * kBox;
// misc: b1 [kMaxF], b2 [D], the broadcast x0 row [D], row statistics
// [sum|var][half][row], barriers, TMEM slot
constexpr uint32_t kMiscB1 = 0;
constexpr uint32_t kMiscB2 = kMiscB1 + kMaxF * 4;
constexpr uint32_t kMiscX0 = kMiscB2 + D * 4;
constexpr uint32_t kMiscRed = kMiscX0 + D * 4;
constexpr uint32_t kMiscBars = kMiscRed + 2 * 2 * 128 * 4;
constexpr uint32_t kMiscBytes = kMiscBars + 32 * 8 + 16;
constexpr size_t kSmem = 1024 + kOffMisc + kMiscBytes;
static_assert(kSmem <= 232448, "shared memory budget");

__device__ __forceinline__ float relu_nan256(float x) {
  float r;
  asm("max.NaN.f32 %0, %1, 0f00000000;" : "=f"(r) : "f"(x));
  return r;
}

__device__ __forceinline__ void arrive_one(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// dst (+)= (k block of the split A tile: hi plane at sa, lo plane at sa + 16 KB)
// . (weight box at w)^T, M = N = 128, K = 64: eight products.
__device__ __noinline__ void mma_box(uint32_t dst, uint32_t sa, uint32_t w, uint32_t idesc, bool acc) {
  const uint32_t go = elect_one();  // (the lane that the caller's commits elect)
  const uint64_t a0 = umma_desc_sw128(sa);
  const uint64_t w0 = umma_desc_sw128(w);
#pragma unroll
  for (int kk = 0; kk < BK / 16; ++kk) {
    const uint64_t ah = desc_adv(a0, kk * 32);
    const uint64_t wh = desc_adv(w0, kk * 32);
    umma_bf16_if(dst, ah, wh, idesc, (acc || kk != 0) ? 1u : 0u, go);
    umma_bf16_if(dst, desc_adv(ah, kBox), wh, idesc, 1u, go);
  }
}

// Row r, columns c .. c + 31 (c a multiple of 32) as a split bf16 pair into
// the A tile [kb][plane] (128-byte swizzle).
__device__ __forceinline__ void store_split_cols(uint8_t* sA, int r, int c, const float* v) {
  uint32_t hi[16], lo[16];
#pragma unroll
  for (int j = 0; j < 16; ++j) split2(v[2 * j], v[2 * j + 1], hi[j], lo[j]);
  uint8_t* rowp = sA + (size_t)((c >> 6) * 2) * kBox + (size_t)r * 128u;
  const int u0 = (c & 63) >> 3;
#pragma unroll
  for (int jj = 0; jj < 4; ++jj) {
    const uint32_t o = (uint32_t)((u0 + jj) ^ (r & 7)) << 4;
    *reinterpret_cast<uint4*>(rowp + o) = make_uint4(hi[4 * jj], hi[4 * jj + 1], hi[4 * jj + 2], hi[4 * jj + 3]);
    *reinterpret_cast<uint4*>(rowp + kBox + o) = make_uint4(lo[4 * jj], lo[4 * jj + 1], lo[4 * jj + 2], lo[4 * jj + 3]);
  }
}
}  // namespace

__global__ void __launch_bounds__(kThreads, 1)
    ffn256_kernel(const __grid_constant__ CUtensorMap tA_h, const __grid_constant__ CUtensorMap tA_l,
                  const __grid_constant__ CUtensorMap tWO, const __grid_constant__ CUtensorMap tW1,
                  const __grid_constant__ CUtensorMap tW2, const __grid_constant__ CUtensorMap tT,
                  const __grid_constant__ CUtensorMap tO_h, const __grid_constant__ CUtensorMap tO_l,
                  const __grid_constant__ CUtensorMap tX, const __grid_constant__ CUtensorMap tQ,
                  const Ffn256Params p) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw_s = smem_u32(smem_raw);
  uint8_t* smem = smem_raw + ((1024u - (raw_s & 1023u)) & 1023u);
  uint8_t* sA = smem;              // the A tile, then LN(x), then LN(x_out) [kb][plane]
  uint8_t* sR = smem + kABytes;    // weight ring [kRing][16 KB]
  uint8_t* misc = smem + kOffMisc;
  float* sB1 = reinterpret_cast<float*>(misc + kMiscB1);
  float* sB2 = reinterpret_cast<float*>(misc + kMiscB2);
  float* sX0 = reinterpret_cast<float*>(misc + kMiscX0);
  float* red = reinterpret_cast<float*>(misc + kMiscRed);
  uint64_t* bars = reinterpret_cast<uint64_t*>(misc + kMiscBars);
  uint64_t* w_full = bars;           // [kRing]
  uint64_t* w_empty = bars + 5;      // [kRing]
  uint64_t* a_full = bars + 24;      // [NKB] k block of the A tile loaded
  uint64_t* a_free = bars + 28;      // [NKB] k block of sA free for the next tile
  uint64_t* o_done = bars + 12;      // A W_O complete
  uint64_t* ln_full = bars + 13;     // x in the accumulator, LN(x) in sA
  uint64_t* acc1_full = bars + 14;   // [2]
  uint64_t* acc1_empty = bars + 16;  // [2]
  uint64_t* mid_full = bars + 18;    // [2]
  uint64_t* acc2_full = bars + 20;   // FFN2 of the tile complete
  uint64_t* tail_a = bars + 21;      // LN(x_out) in sA
  uint64_t* tail_full = bars + 22;   // the tail product complete
  uint64_t* drain = bars + 23;       // the products in flight at the end
  uint64_t* q_read = bars + 10;      // the tail product read
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 32);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int F = p.F, nf = F / FC;
  if (threadIdx.x == 0) {
    for (int i = 0; i < kRing; ++i) {
      mbar_init(w_full + i, 1);
      mbar_init(w_empty + i, 1);
    }
    for (int i = 0; i < NKB; ++i) {
      mbar_init(a_full + i, 1);
      mbar_init(a_free + i, 1);
    }
    mbar_init(q_read, kEpiWarps);
    mbar_init(o_done, 1);
    mbar_init(ln_full, kEpiWarps);
    for (int i = 0; i < 2; ++i) {
      mbar_init(acc1_full + i, 1);
      mbar_init(acc1_empty + i, 1);
      mbar_init(mid_full + i, kEpiWarps);
    }
    mbar_init(acc2_full, 1);
    mbar_init(tail_a, kEpiWarps);
    mbar_init(tail_full, 1);
    mbar_init(drain, 1);
    fence_mbar_init();
    prefetch_tmap(&tA_h);
    prefetch_tmap(&tWO);
    prefetch_tmap(&tW1);
    prefetch_tmap(&tW2);
  }
  // biases and the broadcast row are parameters: read before the dependency wait
  for (int i = threadIdx.x; i < F; i += kThreads) sB1[i] = p.b1[i];
  for (int i = threadIdx.x; i < D; i += kThreads) {
    sB2[i] = p.b2[i];
    sX0[i] = p.x0_row ? p.x0_row[i] : 0.f;
  }
  if (warp == 0) tmem_alloc(tmem_slot, 512);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  const uint32_t acc2 = tmem + 256u;
  pdl_trigger();
  pdl_wait();
  int rows_valid = p.rows;
  if (p.rows_dev) rows_valid = min(*p.rows_dev, p.rows);
  const int tiles = (rows_valid + BM - 1) / BM;

  // Warps 0 and 1 run whole (fe_common.cuh): uniform control flow, the
  // instructions predicated on the elected lane.
  if (warp == 0) {
    // ---------------- TMA producer ----------------
    const uint32_t go = elect_one();
    int slot = 0, tl = 0;
    uint32_t par = 1;  // the parity of the slot's previous release (a fresh barrier passes)
    // every CTA re-reads the same weight boxes while the activation tiles
    // stream past once: keep the weights in L2, let the activations go first
    const uint64_t keep = l2_policy_evict_last(), pass = l2_policy_evict_first();
    auto load = [&](const CUtensorMap* m, int x, int y) {
      mbar_wait_load(w_empty + slot, w_full + slot, par, p.status);
      mbar_arrive_expect_tx_if(w_full + slot, kBox, go);
      tma_load_2d_hint_if(sR + (size_t)slot * kBox, m, x, y, w_full + slot, keep, go);
      if (++slot == kRing) {
        slot = 0;
        par ^= 1u;
      }
    };
    for (int t = blockIdx.x; t < tiles; t += gridDim.x, ++tl) {
      // W_O boxes (kb, nh) in the MMA's order; the first four may load while
      // the previous tile still uses sA
      for (int i = 0; i < 2 * NKB; ++i) {
        if (i == kRing - 1) {
          for (int kb = 0; kb < NKB; ++kb) {
            if (tl > 0) mbar_wait_load(a_free + kb, a_full + kb, (tl - 1) & 1, p.status);
            mbar_arrive_expect_tx_if(a_full + kb, 2 * kBox, go);
            tma_load_2d_hint_if(sA + (size_t)(kb * 2) * kBox, &tA_h, kb * BK, t * BM, a_full + kb, pass, go);
            tma_load_2d_hint_if(sA + (size_t)(kb * 2 + 1) * kBox, &tA_l, kb * BK, t * BM, a_full + kb, pass, go);
          }
        }
        load(&tWO, (i >> 1) * BK, (i & 1) * 128);
      }
      for (int s = 0; s <= nf; ++s) {
        if (s < nf)
          for (int kb = 0; kb < NKB; ++kb) load(&tW1, kb * BK, s * FC);
        if (s >= 1)
          for (int i = 0; i < 4; ++i)  // (nh, sub): sub fastest
            load(&tW2, (s - 1) * FC + (i & 1) * BK, (i >> 1) * 128);
        // the next tile's A and x0 into L2 meanwhile
        if (t + gridDim.x < tiles)
          for (int kb = s; kb < NKB; kb += nf + 1) {
            const int y = (t + gridDim.x) * BM;
            tma_prefetch_2d_if(&tA_h, kb * BK, y, go);
            tma_prefetch_2d_if(&tA_l, kb * BK, y, go);
            if (!p.x0_row)
              for (int i = 0; i < 8; ++i) tma_prefetch_2d_if(&tX, kb * BK + (i & 1) * 32, y + (i >> 1) * 32, go);
          }
      }
      if (p.tail)
        for (int i = 0; i < 2 * NKB; ++i) load(&tT, (i >> 1) * BK, (i & 1) * 128);
    }
    // the last loads land before this block's shared memory goes away (after a
    // timed-out wait nothing else has waited for them)
    mbar_landed_ring(w_full, slot, par, kRing, p.status);
    mbar_landed_ring(a_full, 0, (tl & 1) ^ 1, NKB, p.status);
  } else if (warp == 1) {
    // ---------------- MMA issuer ----------------
    const uint32_t go = elect_one();
    const uint32_t idesc = umma_idesc_bf16(BM, 128);
    int slot = 0, tl = 0, gf = 0;
    uint32_t par = 0;
    auto wait = [&](uint64_t* bar, uint32_t parity) {
      mbar_wait_role(bar, parity, p.status);
      tc_fence_after();
    };
    // the next weight box landed: its shared-memory address
    auto next_box = [&]() -> uint32_t {
      wait(w_full + slot, par);
      return smem_u32(sR + (size_t)slot * kBox);
    };
    // the box's slot frees once the products issued so far complete
    auto release = [&]() {
      umma_commit_if(w_empty + slot, go);
      if (++slot == kRing) {
        slot = 0;
        par ^= 1u;
      }
    };
    // [0, 256) = LN-free product of the A tile in sA with a 256 x 256 weight
    // (W_O or W_Q), box by box: k block kb, output half nh
    // `full`: the k blocks' barriers where the tile may still be landing
    auto mma_256 = [&](uint64_t* full, uint32_t fpar) {
      for (int i = 0; i < 2 * NKB; ++i) {
        const int kb = i >> 1, nh = i & 1;
        if (full && nh == 0) wait(full + kb, fpar);
        const uint32_t w = next_box();
        mma_box(tmem + (uint32_t)(nh * 128), smem_u32(sA) + (uint32_t)(kb * 2) * kBox, w, idesc, kb != 0);
        release();
      }
    };
    for (int t = blockIdx.x; t < tiles; t += gridDim.x, ++tl) {
      // ---- A W_O into [0, 256) (the previous tile's tail product read)
      if (p.tail && tl > 0) wait(q_read, (tl - 1) & 1);
      mma_256(a_full, tl & 1);
      umma_commit_if(o_done, go);
      // ---- FFN1 chunk s one chunk ahead of FFN2 chunk s - 1
      wait(ln_full, tl & 1);
      const int gf0 = gf;
      for (int s = 0; s <= nf; ++s) {
        if (s < nf) {
          const int g = gf0 + s, b = g & 1;
          if (g >= 2) wait(acc1_empty + b, ((g >> 1) - 1) & 1);
          for (int kb = 0; kb < NKB; ++kb) {
            const uint32_t w = next_box();
            mma_box(tmem + (uint32_t)(b * FC), smem_u32(sA) + (uint32_t)(kb * 2) * kBox, w, idesc, kb != 0);
            release();
          }
          umma_commit_if(acc1_full + b, go);
        }
        if (s >= 1) {
          const int c = s - 1, g = gf0 + c, b = g & 1;
          wait(mid_full + b, (g >> 1) & 1);
          // each 32-column piece of the buffer: 32 hidden units as the hi plane
          // (16 columns of bf16 pairs) then the lo plane
          const uint32_t mt = tmem + (uint32_t)(b * FC);
          for (int i = 0; i < 4; ++i) {
            const int nh = i >> 1, sub = i & 1;
            const uint64_t w0 = umma_desc_sw128(next_box());
#pragma unroll
            for (int k4 = 0; k4 < 4; ++k4) {
              const uint32_t mh = mt + (uint32_t)(64 * sub + 32 * (k4 >> 1) + 8 * (k4 & 1)), ml = mh + 16;
              const uint64_t wh = desc_adv(w0, (uint32_t)k4 * 32);
              umma_bf16_tmem_a_if(acc2 + (uint32_t)(nh * 128), mh, wh, idesc, 1u, go);
              umma_bf16_tmem_a_if(acc2 + (uint32_t)(nh * 128), ml, wh, idesc, 1u, go);
            }
            release();
          }
          umma_commit_if(acc1_empty + b, go);
          if (c == nf - 1) umma_commit_if(acc2_full, go);
        }
      }
      gf = gf0 + nf;
      // ---- the tail LN(x_out) W_Q into [0, 256)
      if (p.tail) {
        wait(tail_a, tl & 1);
        mma_256(nullptr, 0);
        umma_commit_if(tail_full, go);
      }
    }
    umma_drain(drain, p.status, go);
  } else {
    // ---------------- epilogue (warps 2..9) ----------------
    // two warps per TMEM lane quadrant q; warp half hf owns columns
    // [128 hf, 128 hf + 128) of the row, as four 32-column pieces
    const int ew = warp - 2, q = warp & 3, hf = ew >> 2;
    const int et = threadIdx.x - 64;
    const int r = q * 32 + lane;
    const uint32_t lane_off = (uint32_t)(q * 32) << 16;
    const int c0 = 128 * hf;
    float* red_sum = red;        // [half][row]
    float* red_var = red + 256;  // [half][row]
    auto pair_sync = [&]() { asm volatile("bar.sync %0, 64;" ::"r"(1 + q) : "memory"); };
    auto half_sync = [&]() { asm volatile("bar.sync %0, 128;" ::"r"(6 + hf) : "memory"); };
    const bool lead = (et & 127) == 0;  // issues its half's stores
    auto epi_sync = [&]() { asm volatile("bar.sync 5, %0;" ::"n"(32 * kEpiWarps) : "memory"); };
    auto warp_arrive = [&](uint64_t* bar) {
      __syncwarp();
      if (lane == 0) arrive_one(bar);
    };
    auto wait = [&](uint64_t* bar, uint32_t par) { mbar_wait_role(bar, par, p.status); };
    // the row statistics over both halves: sum -> mean, then sum of squares -> rstd
    auto pair_mean = [&](float s) {
      red_sum[hf * 128 + r] = s;
      pair_sync();
      return (red_sum[r] + red_sum[128 + r]) * (1.f / (float)D);
    };
    auto pair_rstd = [&](float s) {
      red_var[hf * 128 + r] = s;
      pair_sync();
      return 1.0f / sqrtf((red_var[r] + red_var[128 + r]) * (1.f / (float)D) + p.eps);
    };
    int tl = 0, gf = 0;
    for (int t = blockIdx.x; t < tiles; t += gridDim.x, ++tl) {
      const int m0 = t * BM;
      const bool valid = m0 + r < rows_valid;
      float* xrow = p.x + (size_t)(m0 + r) * p.ldx;
      // ---- x0 into the accumulator while the projection runs (x0 of rows past
      // the valid count is 0)
#pragma unroll 1
      for (int i = 0; i < 4; ++i) {
        const int c = c0 + 32 * i;
        float v[32];
#pragma unroll
        for (int j = 0; j < 32; j += 8) {
#pragma unroll
          for (int i = 0; i < 8; ++i) v[j + i] = p.x0_row ? sX0[c + j + i] : 0.f;
          if (!p.x0_row && valid) ld_sector(xrow + c + j, v + j);
        }
        tmem_st32(acc2 + lane_off + (uint32_t)c, v);
      }
      // ---- x = x0 + A W_O back into the accumulator, LN(x) over the A tile
      // (the projection, the tile's only reader, is complete)
      wait(o_done, tl & 1);
      tc_fence_after();
      RowSum sum0, var0;
#pragma unroll 1
      for (int i = 0; i < 4; ++i) {
        const int c = c0 + 32 * i;
        float v[32], w[32];
        tmem_ld32(tmem + lane_off + (uint32_t)c, v);
        tmem_ld32(acc2 + lane_off + (uint32_t)c, w);
        row_plus<32>(v, w);
        row_add<32>(sum0, v);
        tmem_st32(acc2 + lane_off + (uint32_t)c, v);
      }
      const float mean0 = pair_mean(sum0.total());
#pragma unroll 1
      for (int i = 0; i < 4; ++i) {
        float v[32];
        tmem_ld32(acc2 + lane_off + (uint32_t)(c0 + 32 * i), v);
        row_add_sq<32>(var0, v, mean0);
      }
      const float rstd0 = pair_rstd(var0.total());
#pragma unroll 1
      for (int i = 0; i < 4; ++i) {
        const int c = c0 + 32 * i;
        float v[32];
        tmem_ld32(acc2 + lane_off + (uint32_t)c, v);
        row_norm<32>(v, mean0, rstd0);
        store_split_cols(sA, r, c, v);
      }
      fence_async_shared();
      tc_fence_before();
      warp_arrive(ln_full);
      // ---- per chunk: split(ReLU(acc1 + b1)) over this thread's 64 columns of
      // the chunk's TMEM buffer, FFN2's A operand
      for (int f = 0; f < nf; ++f, ++gf) {
        const int ba = gf & 1;
        wait(acc1_full + ba, (gf >> 1) & 1);
        tc_fence_after();
#pragma unroll 1
        for (int jp = 0; jp < 2; ++jp) {
          const uint32_t col = tmem + lane_off + (uint32_t)(ba * FC + 64 * hf + 32 * jp);
          const float* bias = sB1 + f * FC + 64 * hf + 32 * jp;
          float v[32];
          tmem_ld32(col, v);
          uint32_t hi[16], lo[16];
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            const float2 bb = *reinterpret_cast<const float2*>(bias + 2 * j);
            const float b2[2] = {bb.x, bb.y};
            row_plus<2>(v + 2 * j, b2);
            split2_trunc(relu_nan256(v[2 * j]), relu_nan256(v[2 * j + 1]), hi[j], lo[j]);
          }
          tmem_st16_nowait(col, hi);
          tmem_st16_nowait(col + 16u, lo);
        }
        tmem_st_wait();
        tc_fence_before();
        warp_arrive(mid_full + ba);
      }
      // ---- x_out = acc2 + b2 to memory, staged in this warp's 16 KB of sA (every
      // FFN1 has read LN(x) there) as four 32 x 32 blocks (128-byte swizzle)
      // and stored by TMA; then LN(x_out) over the A tile
      wait(acc2_full, tl & 1);
      tc_fence_after();
      uint8_t* xst = sA + (size_t)ew * 16384u;
      RowSum sum, var;
#pragma unroll 1
      for (int i = 0; i < 4; ++i) {
        const int c = c0 + 32 * i;
        float v[32];
        tmem_ld32(acc2 + lane_off + (uint32_t)c, v);
        uint8_t* blk = xst + (size_t)i * 4096u + (uint32_t)lane * 128u;
#pragma unroll
        for (int j = 0; j < 32; j += 4) {
          const float4 bb = *reinterpret_cast<const float4*>(sB2 + c + j);
          const float b4[4] = {bb.x, bb.y, bb.z, bb.w};
          row_plus<4>(v + j, b4);
          row_add<4>(sum, v + j);
          *reinterpret_cast<float4*>(blk + ((uint32_t)((j >> 2) ^ (lane & 7)) << 4)) =
              make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]);
        }
      }
      fence_async_shared();
      __syncwarp();
      if (lane == 0) {
        for (int i = 0; i < 4; ++i) tma_store_2d(&tX, xst + (size_t)i * 4096u, c0 + 32 * i, m0 + 32 * q);
        bulk_commit();
      }
      const float mean = pair_mean(sum.total());
#pragma unroll 1
      for (int i = 0; i < 4; ++i) {
        const int c = c0 + 32 * i;
        float v[32];
        tmem_ld32(acc2 + lane_off + (uint32_t)c, v);
#pragma unroll
        for (int j = 0; j < 32; j += 4) {
          const float4 bb = *reinterpret_cast<const float4*>(sB2 + c + j);
          const float b4[4] = {bb.x, bb.y, bb.z, bb.w};
          row_plus<4>(v + j, b4);
          row_add_sq<4>(var, v + j, mean);
        }
      }
      const float rstd = pair_rstd(var.total());
      if (lane == 0) bulk_wait_read0();
      epi_sync();  // every warp's x_out staging read: sA takes LN(x_out)
#pragma unroll 1
      for (int i = 0; i < 4; ++i) {
        const int c = c0 + 32 * i;
        float v[32];
        tmem_ld32(acc2 + lane_off + (uint32_t)c, v);
#pragma unroll
        for (int j = 0; j < 32; j += 4) {
          const float4 bb = *reinterpret_cast<const float4*>(sB2 + c + j);
          const float b4[4] = {bb.x, bb.y, bb.z, bb.w};
          row_plus<4>(v + j, b4);
          row_norm<4>(v + j, mean, rstd);
        }
        store_split_cols(sA, r, c, v);
        if (i & 1) {
          fence_async_shared();
          if (p.store_ln) {
            half_sync();  // every row of k block c / 64 written
            if (lead) {
              const int kb = c >> 6;
              tma_store_2d(&tO_h, sA + (size_t)(kb * 2) * kBox, kb * BK, m0);
              tma_store_2d(&tO_l, sA + (size_t)(kb * 2 + 1) * kBox, kb * BK, m0);
              bulk_commit();
            }
            __syncwarp();
          }
        }
      }
      tc_fence_before();
      if (p.tail) {
        // ---- the tail: Q = LN(x_out) W_Q as f16 over the upper half of sA (the
        // tail product has read LN(x_out), whose stores have read it too): this
        // thread's 128 columns of row r as 128-byte-swizzled [kb][128 rows x 64]
        // tiles, stored by TMA
        warp_arrive(tail_a);
        wait(tail_full, tl & 1);
        tc_fence_after();
        if (p.store_ln) {
          if (lead) bulk_wait_read0();
          epi_sync();
        }
        if (et == 0) {
          arrive_one(a_free);
          arrive_one(a_free + 1);
        }
        __syncwarp();
        uint8_t* sQ = sA + (size_t)4 * kBox;
#pragma unroll 1
        for (int i = 0; i < 4; ++i) {
          const int c = c0 + 32 * i;
          float v[32];
          tmem_ld32(tmem + lane_off + (uint32_t)c, v);
          uint8_t* rowp = sQ + (size_t)(c >> 6) * kBox + (size_t)r * 128u;
          const int u0 = (c & 63) >> 3;
#pragma unroll
          for (int j = 0; j < 4; ++j)
            *reinterpret_cast<uint4*>(rowp + ((uint32_t)((u0 + j) ^ (r & 7)) << 4)) =
                make_uint4(pack_f16x2(v[8 * j], v[8 * j + 1]), pack_f16x2(v[8 * j + 2], v[8 * j + 3]),
                           pack_f16x2(v[8 * j + 4], v[8 * j + 5]), pack_f16x2(v[8 * j + 6], v[8 * j + 7]));
        }
        tc_fence_before();
        warp_arrive(q_read);
        fence_async_shared();
        half_sync();  // every row of this half's Q written
        if (lead) {
          for (int kb = 2 * hf; kb < 2 * hf + 2; ++kb) tma_store_2d(&tQ, sQ + (size_t)kb * kBox, kb * BK, m0);
          bulk_commit();
          bulk_wait_read0();
          arrive_one(a_free + 2 + hf);
        }
      } else {
        // ---- a k block may take the next tile's A once its store has read it
        // (the TMEM columns [0, 256) were last read before the FFN2 products)
        if (!p.store_ln) half_sync();
        if (lead) {
          bulk_wait_read1();
          arrive_one(a_free + 2 * hf);
          bulk_wait_read0();
          arrive_one(a_free + 2 * hf + 1);
        }
      }
      __syncwarp();
    }
    if (lane == 0) bulk_wait0();  // output tensor stores complete before the CTA retires
  }

  __syncwarp();
  tc_fence_before();
  __syncthreads();
  if (warp == 0) tmem_dealloc(tmem, 512);
}

namespace {
int g_ffn256_sms = 0;
}

bool ffn256_supported(int d, int F, int nb) { return d == D && nb == 1 && F % FC == 0 && F >= FC && F <= kMaxF; }

cudaError_t ffn256_prepare() {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&g_ffn256_sms, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(ffn256_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem);
  return e;
}

cudaError_t ffn256_launch(const CUtensorMap* a_h, const CUtensorMap* a_l, const CUtensorMap* wo, const CUtensorMap* w1,
                          const CUtensorMap* w2, const CUtensorMap* wt, const CUtensorMap* o_h, const CUtensorMap* o_l,
                          const CUtensorMap* x_st, const CUtensorMap* q_st, const Ffn256Params& p, cudaStream_t s) {
  if (p.rows <= 0) return cudaSuccess;
  if (!ffn256_supported(D, p.F, 1) || !x_st || (p.tail && !wt) || (p.tail && !q_st)) return cudaErrorInvalidValue;
  if (!p.x0_row && (p.ldx % 8 || (uintptr_t)p.x % 32)) return cudaErrorInvalidValue;  // (ld_sector)
  const long long tiles = (p.rows + BM - 1) / BM;
  long long grid = g_ffn256_sms > 0 ? g_ffn256_sms : 148;
  if (grid > tiles) grid = tiles;
  return launch_k(ffn256_kernel, dim3((unsigned)grid), dim3(kThreads), kSmem, s, *a_h, *a_l, *wo, *w1, *w2,
                  p.tail ? *wt : *wo, *o_h, *o_l, *x_st, p.tail ? *q_st : *o_h, p);
}

}  // namespace fe
