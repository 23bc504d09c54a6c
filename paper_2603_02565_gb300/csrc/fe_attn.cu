// Flash-style multi-head attention over request segments, on tcgen05.
//
// Used twice in the evaluator:
//  * element -> context cross-attention (Section 4.2): the query rows are the
//    distinct elements of request b, the keys/values its C context rows, so
//    the context K/V computed once per request serve every element;
//  * cross-sequence self-attention (Section 4.4) over the K sequence vectors.
//
// One persistent CTA per SM holds independent groups (four with 64-key chunks
// for d_h = 32, two with 128-key chunks for d_h = 64), each walking its own
// units (segment, head, 128-row query tile):
//   warp g (role)  : group g's loads (TMA; Q tile and a ring of K/V chunks)
//                    and its tcgen05.mma: S_{j+1} = Q K_{j+1}^T as soon as the
//                    softmax has S_j in registers, PV_j = P_j V_j once P_j is
//                    written, accumulated in TMEM over the unit
//   4 warps        : softmax, one query row and all keys of the chunk per
//                    lane, so that nothing is exchanged between threads;
//                    P_j goes to TMEM as f16 against a running maximum that
//                    moves only when a chunk exceeds it by more than 8 (log2
//                    units), when the output accumulator is rescaled
// TMEM per group: S, P (half as many columns), the output accumulator (d_h).
//
// What bounds it: the softmax's issue slots and exponents and, at these narrow
// shapes, the tensor pipe about equally (per 128 x 64 chunk: 64 exponents a
// lane at 4 cycles a warp, six MMAs of N <= 64 at 40-48 cycles), if enough
// warps are in flight; hence one softmax warp of every group on every SM
// sub-partition.  A warp can only read the TMEM lanes of its own sub-partition,
// so a tile with fewer than 97 rows leaves some of them idle: group g places
// row block k of a tile in lane quadrant (k - g) mod 4, which spreads the idle
// ones.  The scaling and the sums use two-element fp32 instructions.
// Measured against one unit per CTA, two CTAs per SM, eight softmax warps a unit
// (two per lane quadrant, exchanging row maxima) and units dealt out tile by tile:
// 1024 requests x 512 keys x 8 heads 811 -> 435 us a launch, K = 1000 cross-sequence
// attention 103 -> 95, the two of 256 requests 42 -> 41.  A lone
// unit (one request) takes about 2 us longer than with eight warps, and more the
// longer its keys, so from 32 chunks on idle groups share it (SPLIT).  The softmax of
// four groups still takes about 2300 cycles a chunk where the same instructions
// without barriers take 1400: latency between the roles, not a pipe.
// Register split: the kernel's arithmetic keeps a chunk's 64 (128) scores per lane
// in registers, so the softmax warps take registers from the role warps
// (setmaxnreg; without it spills cost 2 to 4 %).
// Q, K, V and P are single f16 planes (unit roundoff 2^-11; Q and K come
// from LayerNorm'd rows times weights of magnitude well inside the f16
// range, P lies in [0, 2^8]); accumulation, softmax statistics and the output
// are fp32, the output leaves as a bf16 hi/lo pair.
#include "fe_common.cuh"
#include "fe_kernels.h"

namespace fe {

namespace {

constexpr int BQ = 128;     // query rows per unit (TMEM lanes)
constexpr int kRoleWarps = 4;

template <int DH>
struct AttnCfg {
  static constexpr int NG = DH == 32 ? 4 : 2;                   // groups per CTA
  static constexpr int CK = DH == 32 ? 64 : 128;                // keys per chunk
  static constexpr int kThreads = 32 * (kRoleWarps + 4 * NG);
  // TMEM per group: S at [0, CK), P at [CK, 3 CK / 2), then the output accumulator
  static constexpr int kP = CK, kO = CK + CK / 2;
  static constexpr int kGroupCols = kO + DH;
  static_assert(NG * kGroupCols <= 512, "TMEM budget");
  static constexpr uint32_t kRowBytes = DH * 2;                 // one row of a Q/K/V tile
  static constexpr uint32_t kQBlock = 32 * kRowBytes;           // Q rows of one lane quadrant
  static constexpr uint32_t kQBytes = 4 * kQBlock;              // Q tile: 128 rows
  static constexpr uint32_t kKVTile = CK * kRowBytes;           // K or V chunk
  static constexpr uint32_t kKVBytes = 2 * kKVTile;             // K, V
  static constexpr uint32_t kSwz = DH == 32 ? 4u : 2u;          // descriptor swizzle code (64 B / 128 B)
  static constexpr uint32_t kSbo = 8 * kRowBytes;               // 8-row swizzle atom
  static constexpr int NQ = 2;                                  // Q buffers (and the unit's output staging)
  static constexpr int NS = DH == 32 ? 5 : 2;                   // K/V stages (at least 2)
  static constexpr bool kLoader = NG <= 2;                      // a warp of its own for the loads of a group
  static constexpr uint32_t kGroupBytes = NQ * kQBytes + NS * kKVBytes;
  static constexpr int NC = DH / 8;                             // 16-byte pieces of a row
  // staging piece of row `row`: XOR mask (eight consecutive 16-byte accesses on distinct banks)
  __device__ static constexpr uint32_t swz(int row) { return NC == 8 ? (row & 7) : ((row >> 1) & 3); }
  static constexpr int kBars = NQ + 2 * NS + 4;                 // mbarriers per group
  static constexpr size_t kSmem = 1024 + NG * (size_t)kGroupBytes + NG * kBars * 8 + 64;
  static_assert(kSmem <= 232448, "shared memory budget");
};

__device__ __forceinline__ uint64_t desc_sw(uint32_t saddr, uint32_t sbo, uint32_t swz) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);
  d |= (uint64_t)1 << 16;                       // leading byte offset (unused: one atom wide)
  d |= (uint64_t)(sbo >> 4) << 32;              // stride byte offset: next 8-row atom
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)swz << 61;
  return d;
}

__device__ __forceinline__ float max3f(float a, float b, float c) {
  float r;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}

// maximum of N values: four chains of three-input maxima (few live registers)
template <int N>
__device__ __forceinline__ float maxn(const float* v) {
  float a[4] = {v[0], v[1], v[2], v[3]};
#pragma unroll
  for (int i = 4; i + 8 <= N; i += 8) {
#pragma unroll
    for (int k = 0; k < 4; ++k) a[k] = max3f(a[k], v[i + 2 * k], v[i + 2 * k + 1]);
  }
#pragma unroll
  for (int k = 0; k < 2; ++k) a[k] = max3f(a[k], v[N - 4 + 2 * k], v[N - 3 + 2 * k]);  // N % 8 == 0
  return fmaxf(max3f(a[0], a[1], a[2]), a[3]);
}

// Work of a group.  The W = sb * n_heads * tp groups of the grid that have work
// are numbered (query tile offset, segment, head), head fastest; in one round
// they take tiles t .. t + tp - 1 of sb consecutive segments, all heads, in the
// next one the following tiles of the same segments, then the next sb segments.
// Every group thus gets the same tile index in the same round, whatever the
// segments' row counts (the last tiles are short or empty: with units dealt out
// tile by tile the group stride was a multiple of the tile count, and the SMs that
// drew the last tile stood idle: 43 % of the SM time at 290 of 500 rows), and
// the tiles of a segment follow one another while its K/V are in L2.
// The segment count and offset of the next segment are loaded one segment
// ahead, so that moving to it does not wait on a global load.
struct Cursor {
  int b, q0, qcnt, qoff;  // segment (n_segments and more: no work left), tile row, its rows and offset
  int ncnt, noff;         // q_cnt / q_off of segment b + sb
};

// rows and offset of segment b (none past the last), this lane's copy
__device__ __forceinline__ void seg_load(const AttnParams& p, int b, int& cnt, int& off) {
  const bool in = b < p.n_segments;
  cnt = !in ? 0 : p.q_cnt_dev ? __ldg(p.q_cnt_dev + b) : p.q_cnt_fixed;
  off = !in ? 0 : p.q_off_dev ? __ldg(p.q_off_dev + b) : b * p.q_stride;
}
// (every lane of a warp holds the cursor; the broadcast makes the loaded
// values, and the control flow that follows from them, uniform)
__device__ __forceinline__ int warp_value(int v) { return __shfl_sync(0xffffffffu, v, 0); }

// from a segment whose tiles are done to the next one with rows at the group's first tile
__device__ __forceinline__ void cur_segment(const AttnParams& p, int first_row, Cursor& c) {
  while (c.b < p.n_segments && c.q0 >= c.qcnt) {
    c.b += p.sb;
    c.q0 = first_row;
    c.qcnt = c.ncnt;
    c.qoff = c.noff;
    int cnt, off;
    seg_load(p, c.b + p.sb, cnt, off);
    c.ncnt = warp_value(cnt);
    c.noff = warp_value(off);
  }
}

__device__ __forceinline__ void cur_first(const AttnParams& p, int b0, int first_row, Cursor& c) {
  int cnt, off, cnt2, off2;  // the four loads together: one memory latency
  seg_load(p, b0, cnt, off);
  seg_load(p, b0 + p.sb, cnt2, off2);
  c = Cursor{b0, first_row, warp_value(cnt), warp_value(off), warp_value(cnt2), warp_value(off2)};
  cur_segment(p, first_row, c);
}

__device__ __forceinline__ void cur_next(const AttnParams& p, int first_row, Cursor& c) {
  c.q0 += p.tp * BQ;
  cur_segment(p, first_row, c);
}

// Zero bytes [o0, end) of a shared-memory tile (one warp, 16-byte stores),
// then order the writes before the warp's next tensor-core operations.
__device__ __forceinline__ void zero_tail(uint8_t* t, int o0, int end) {
  for (int o = o0 + 16 * (int)(threadIdx.x & 31); o < end; o += 512)
    *reinterpret_cast<uint4*>(t + o) = make_uint4(0u, 0u, 0u, 0u);
  fence_async_shared();
  __syncwarp();
}

}  // namespace

// SPLIT: p.ks groups of a CTA take one unit together (the only one of each of them),
// group grp its chunks [part kper, (part + 1) kper), part = grp % ks, none of them
// empty; their outputs, each against its own maximum, are put together at the end
// through shared memory.
template <int DH, bool SPLIT>
__global__ void __launch_bounds__(AttnCfg<DH>::kThreads, 1)
    attn_kernel(const __grid_constant__ CUtensorMap tQ, const __grid_constant__ CUtensorMap tK,
                const __grid_constant__ CUtensorMap tV, const AttnParams p) {
  using Cfg = AttnCfg<DH>;
  constexpr int NG = Cfg::NG, CK = Cfg::CK, NQ = Cfg::NQ, NS = Cfg::NS, NC = Cfg::NC;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw_s = smem_u32(smem_raw);
  uint8_t* smem = smem_raw + ((1024u - (raw_s & 1023u)) & 1023u);
  uint64_t* bars0 = reinterpret_cast<uint64_t*>(smem + (size_t)NG * Cfg::kGroupBytes);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars0 + NG * Cfg::kBars);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // group of this warp: role warps (issuers 0 .. NG - 1, then the loaders, if
  // any), then four softmax warps each
  const int grp = warp < kRoleWarps ? warp % NG : (warp - kRoleWarps) >> 2;
  const int j0 = SPLIT ? grp % p.ks * p.kper : 0;  // this group's first chunk of a unit
  // keys of a unit's segment: a fixed count at a fixed stride, or, for
  // self-attention within segments, the segment's own query rows
  auto kv_count = [&](const Cursor& c) { return p.kv_self ? c.qcnt : p.kv_cnt; };
  auto kv_base = [&](const Cursor& c) { return p.kv_self ? c.qoff : c.b * p.kv_stride; };
  auto chunks = [&](const Cursor& c) {  // of this group
    const int n = (kv_count(c) + CK - 1) / CK;
    return SPLIT ? min(p.kper, n - j0) : n;
  };

  uint8_t* sQ = smem + (size_t)grp * Cfg::kGroupBytes;  // [NQ][lane quadrant][32 rows]
  uint8_t* sKV = sQ + NQ * Cfg::kQBytes;                // [NS][K, V]
  uint64_t* bars = bars0 + grp * Cfg::kBars;
  uint64_t* q_full = bars;                // [NQ] each softmax warp's rows of the Q tile landed
  uint64_t* kv_full = q_full + NQ;        // [NS]
  uint64_t* kv_empty = kv_full + NS;      // [NS] PV_j (and everything issued before it) complete
  uint64_t* s_full = kv_empty + NS;       // S_j complete
  uint64_t* s_read = s_full + 1;          // S_j in the softmax's registers
  uint64_t* p_full = s_full + 2;          // P_j written
  uint64_t* drain = s_full + 3;           // the issuer's products after a timed-out wait
  if (threadIdx.x < NG) {
    uint64_t* b = bars0 + threadIdx.x * Cfg::kBars;
    const int sr = NQ + 2 * NS + 1;  // q_full, s_read and p_full: one arrival per softmax warp
    for (int i = 0; i < Cfg::kBars; ++i) mbar_init(b + i, (i < NQ || i == sr || i == sr + 1) ? 4u : 1u);
    fence_mbar_init();
  }
  if (threadIdx.x == 0) {
    prefetch_tmap(&tQ);
    prefetch_tmap(&tK);
    prefetch_tmap(&tV);
  }
  if (warp == 0) tmem_alloc(tmem_slot, 512);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot + (uint32_t)(grp * Cfg::kGroupCols);
  // the group's head, first segment (none: past the last) and first tile's row
  const int wi = (SPLIT ? grp / p.ks : grp) * (int)gridDim.x + (int)blockIdx.x;
  const int head = wi % p.n_heads;
  const int b0 = wi < p.sb * p.n_heads * p.tp ? (wi / p.n_heads) % p.sb : p.n_segments;
  const int row0 = wi / (p.n_heads * p.sb) * BQ;
  // the set-up above reads nothing written by earlier kernels; from here on
  // the segment offsets, counts and operands are
  pdl_trigger();
  pdl_wait();

  if (warp < kRoleWarps) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(DH == 32 ? 64 : 80));
    // The chunks of all the group's units form one stream g = 0, 1, ...
    const uint32_t go = elect_one();
    const bool load = !Cfg::kLoader || warp >= NG, issue = warp < NG;
    // loads: unit cursor, chunks loaded of the unit and of all, the unit's chunks, the next stage and its parity
    Cursor lc;
    int lj = 0, l_n = 0, lg = 0, ls = 0;
    uint32_t lpar = 1;
    cur_first(p, b0, row0, lc);
    l_n = chunks(lc);
    auto load_next = [&]() {
      mbar_wait_load(kv_empty + ls, kv_full + ls, lpar, p.status);
      uint8_t* kv = sKV + ls * Cfg::kKVBytes;
      const int row = kv_base(lc) + (j0 + lj) * CK;
      mbar_arrive_expect_tx_if(kv_full + ls, Cfg::kKVBytes, go);
      if (p.kv3d) {  // head-major K/V: one contiguous block per head
        tma_load_3d_if(kv, &tK, 0, row, (p.k_col + head * DH) / DH, kv_full + ls, go);
        tma_load_3d_if(kv + Cfg::kKVTile, &tV, 0, row, (p.v_col + head * DH) / DH, kv_full + ls, go);
      } else {
        tma_load_2d_if(kv, &tK, p.k_col + head * DH, row, kv_full + ls, go);
        if (p.kv_seg)  // rows past the segment's kv_cnt keys are outside the map: zeros
          tma_load_3d_if(kv + Cfg::kKVTile, &tV, p.v_col + head * DH, (j0 + lj) * CK, lc.b, kv_full + ls, go);
        else
          tma_load_2d_if(kv + Cfg::kKVTile, &tV, p.v_col + head * DH, row, kv_full + ls, go);
      }
      ++lg;
      if (++ls == NS) {
        ls = 0;
        lpar ^= 1u;
      }
      if (++lj == l_n) {
        lj = 0;
        cur_next(p, row0, lc);
        l_n = chunks(lc);
      }
    };
    if (issue) {
      // ---------------- MMA issue of group grp (and its loads, unless another warp has them) ----------------
      const uint32_t idesc_s = umma_idesc_f16(BQ, CK);
      const uint32_t idesc_pv = umma_idesc_f16(BQ, DH) | (1u << 16);  // B (V) is MN-major
      // only a variable key count or one that is not a multiple of CK leaves a
      // partial chunk, whose V rows a segmented map already reads as zeros
      const bool pad_v = p.kv_self || (p.kv_cnt % CK != 0 && !p.kv_seg);
      const uint64_t qd0 = desc_sw(smem_u32(sQ), Cfg::kSbo, Cfg::kSwz);
      const uint64_t kd0 = desc_sw(smem_u32(sKV), Cfg::kSbo, Cfg::kSwz);
      const uint64_t vd0 = desc_sw(smem_u32(sKV + Cfg::kKVTile), Cfg::kSbo, Cfg::kSwz);
      // S: the next S's unit, chunk, chunk count, stage, Q buffer; S issued
      Cursor sc = lc;
      int sj = 0, s_nch = l_n, ss = 0, sq = 0, g_s = 0;
      uint32_t spar = 0, sqpar = 0;
      // request chunks up to number `last`, one at a call while the ring first fills, then two
      auto fill = [&](int last) {
        if (Cfg::kLoader) return;
        for (int k = lg < NS ? 1 : 0; k < 2 && lg <= last && lc.b < p.n_segments; ++k) load_next();
      };
      // S of the next chunk, once the softmax holds the previous one
      auto issue_s = [&]() {
        if (sc.b >= p.n_segments) return;
        if (g_s > 0) mbar_wait_role(s_read, (uint32_t)(g_s - 1) & 1u, p.status);
        if (sj == 0) mbar_wait_role(q_full + sq, sqpar, p.status);
        mbar_wait_role(kv_full + ss, spar, p.status);
        tc_fence_after();
        const uint64_t qd = qd0 + (uint64_t)((sq * Cfg::kQBytes) >> 4);
        const uint64_t kd = kd0 + (uint64_t)((ss * Cfg::kKVBytes) >> 4);
#pragma unroll
        for (int kk = 0; kk < DH / 16; ++kk)
          umma_bf16_if(tmem, qd + (uint64_t)(kk * 2), kd + (uint64_t)(kk * 2), idesc_s, kk != 0 ? 1u : 0u, go);
        umma_commit_if(s_full, go);
        // The V rows of a partial chunk past the key count belong to the next
        // segment: their P is 0, but 0 x NaN is NaN, so they are zeroed here
        // (the chunk has landed; its PV, issued later by this warp, reads them)
        if (pad_v) {
          const int kval = kv_count(sc) - (j0 + sj) * CK;
          if (kval < CK) zero_tail(sKV + ss * Cfg::kKVBytes + Cfg::kKVTile, kval * (int)Cfg::kRowBytes, (int)Cfg::kKVTile);
        }
        ++g_s;
        if (++ss == NS) {
          ss = 0;
          spar ^= 1u;
        }
        if (++sj == s_nch) {  // every S of this unit issued
          if (++sq == NQ) {
            sq = 0;
            sqpar ^= 1u;
          }
          sj = 0;
          cur_next(p, row0, sc);
          s_nch = chunks(sc);
        }
      };
      fill(0);
      issue_s();
      bool first = true;  // PV_g opens its unit
      int ps = 0;         // its stage
      for (int g = 0; g < g_s; ++g) {
        const bool next_first = sj == 0;  // S_{g+1} opens a unit
        fill(g - 1 + NS);                 // up to the stage of PV_{g-1}, complete before P_g may be written
        issue_s();                        // S_{g+1}
        mbar_wait_role(p_full, (uint32_t)g & 1u, p.status);
        tc_fence_after();
        const uint64_t vd = vd0 + (uint64_t)((ps * Cfg::kKVBytes) >> 4);
#pragma unroll
        for (int kk = 0; kk < CK / 16; ++kk)
          umma_bf16_tmem_a_if(tmem + (uint32_t)Cfg::kO, tmem + (uint32_t)(Cfg::kP + 8 * kk),
                              vd + (uint64_t)((kk * 16 * Cfg::kRowBytes) >> 4), idesc_pv, (kk != 0 || !first) ? 1u : 0u,
                              go);
        umma_commit_if(kv_empty + ps, go);
        if (++ps == NS) ps = 0;
        first = next_first;
      }
      umma_drain(drain, p.status, go);
    } else if (load) {
      while (lc.b < p.n_segments) load_next();
    }
    // the last loads land before this block's shared memory goes away (after a
    // timed-out wait nothing else has waited for them)
    if (load) mbar_landed_ring(kv_full, ls, lpar, NS, p.status);
  } else {
    // ---------------- softmax / output ----------------
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(DH == 32 ? 104 : 208));
    const int q4 = warp & 3;                     // TMEM lane quadrant
    const int r = ((q4 + grp) & 3) * 32 + lane;  // query row of the tile
    const uint32_t t_s = tmem + ((uint32_t)(q4 * 32) << 16);
    const uint32_t t_p = t_s + (uint32_t)Cfg::kP, t_o = t_s + (uint32_t)Cfg::kO;
    const uint32_t go = elect_one();
    const uint32_t bb = smem_u32(bars);  // the group's barriers
    int u = 0;  // the unit; its Q buffer is u % NQ, and this warp's rows of it take the unit's output
    constexpr uint32_t kKVE = 8u * (NQ + NS), kSFull = 8u * (NQ + 2 * NS);
    const float sc = p.scale_log2;
    int g = 0, ps = 0;         // chunk of the group's stream; the stage of chunk g - 1
    uint32_t ppar = 0;         // the parity of its PV
    // This warp loads its own 32 rows of each unit's Q tile, one unit ahead:
    // row block k of the tile goes to lane quadrant (k - grp) mod 4.  The buffer's
    // previous unit is done with here (its S are complete, its output is stored).
    auto load_q = [&](const Cursor& c, int v) {
      if (c.b >= p.n_segments) return;
      const int buf = v % NQ;
      mbar_landed_at(bb + 8u * (uint32_t)buf, (uint32_t)(v / NQ - 1) & 1u, p.status);  // (a fresh barrier passes)
      const int blk = c.q0 + (r & ~31);
      if (blk < c.qcnt) {
        mbar_arrive_expect_tx_if(q_full + buf, Cfg::kQBlock, go);
        tma_load_2d_if(sQ + buf * Cfg::kQBytes + q4 * Cfg::kQBlock, &tQ, p.q_col + head * DH, c.qoff + blk, q_full + buf,
                       go);
      } else {
        mbar_arrive_if_at(bb + 8u * (uint32_t)buf, go);
      }
    };
    // SPLIT: a group's output of tile row r (16-byte pieces XOR-swizzled) and its maximum and sum, in
    // its K/V stages (every product has read them), and the barrier of the groups that share a unit
    auto part_row = [&](int g2, int k) {
      return smem + (size_t)g2 * Cfg::kGroupBytes + NQ * Cfg::kQBytes + r * (DH * 4) + ((k ^ (r & 7)) << 4);
    };
    auto part_ml = [&](int g2) {
      return reinterpret_cast<float2*>(smem + (size_t)g2 * Cfg::kGroupBytes + NQ * Cfg::kQBytes + BQ * DH * 4) + r;
    };
    auto set_sync = [&]() { asm volatile("bar.sync %0, %1;" ::"r"(1 + grp / p.ks), "r"(128 * p.ks) : "memory"); };
    Cursor c, next;
    cur_first(p, b0, row0, next);
    load_q(next, 0);
    for (c = next; c.b < p.n_segments; c = next) {
      cur_next(p, row0, next);
      load_q(next, u + 1);
      // the running maximum m that P is taken against moves only when a chunk's
      // maximum exceeds it by more than kSlack (log2 units; P <= 2^kSlack stays
      // far inside f16), and then the unit's output accumulator in TMEM is
      // rescaled: most chunks need no correction at all
      constexpr float kSlack = 8.f;
      float m = -INFINITY, l[2] = {0.f, 0.f};
      // a warp whose 32 query rows all lie past the segment's end only keeps
      // the barrier protocol; those rows of P and of the output are never used
      const bool active = c.q0 + (r & ~31) < c.qcnt;
      const int nch = chunks(c);
      for (int j = 0; j < nch; ++j, ++g) {
        mbar_wait_at(bb + kSFull, (uint32_t)g & 1u, p.status);
        if (!active) {
          mbar_arrive_if_at(bb + kSFull + 8u, go);
          if (g > 0) mbar_wait_at(bb + kKVE + 8u * (uint32_t)ps, ppar, p.status);  // one arrival per chunk on p_full
          mbar_arrive_if_at(bb + kSFull + 16u, go);
        } else {
          tc_fence_after();
          float v[CK];
#pragma unroll
          for (int i = 0; i < CK; i += 64) tmem_ld64(t_s + (uint32_t)i, v + i);
          tc_fence_before();
          __syncwarp();
          mbar_arrive_if_at(bb + kSFull + 8u, go);
          // keys past kv_cnt take no part: -inf gives them P = 0
          const int kvalid = kv_count(c) - (j0 + j) * CK;
          if (kvalid < CK) {
#pragma unroll
            for (int i = 0; i < CK; ++i)
              if (i >= kvalid) v[i] = -INFINITY;
          }
          const float mx = maxn<CK>(v) * sc;
          bool pv_done = false;  // PV_{g-1} waited for
          if (j == 0) {
            m = mx;  // the unit's first PV overwrites the accumulator
          } else {
            const bool up = mx > m + kSlack;
            if (__any_sync(0xffffffffu, up)) {
              // the accumulator holds PV up to chunk g - 1: scale it (and l) to the new maximum
              mbar_wait_at(bb + kKVE + 8u * (uint32_t)ps, ppar, p.status);
              pv_done = true;
              tc_fence_after();
              const float corr = up ? ex2_approx(m - mx) : 1.f;
              if (up) m = mx;
              l[0] *= corr;
              l[1] *= corr;
#pragma unroll 1
              for (int o0 = 0; o0 < DH; o0 += 8) {
                uint32_t o[8];
                tmem_ld8(t_o + (uint32_t)o0, o);
#pragma unroll
                for (int i = 0; i < 8; ++i) o[i] = __float_as_uint(__uint_as_float(o[i]) * corr);
                tmem_st8_nowait(t_o + (uint32_t)o0, o);
              }
            }
          }
          // P's columns are free once PV_{g-1} has read them
          if (g > 0 && !pv_done) mbar_wait_at(bb + kKVE + 8u * (uint32_t)ps, ppar, p.status);
          tc_fence_after();
          // P = 2^(s * scale - m) as f16: keys 2c, 2c+1 in column c
          const uint64_t sc2 = f32x2_pack(sc, sc), nm2 = f32x2_pack(-m, -m);
          // (the two halves of the chunk are summed apart, each in four partial sums of key pairs)
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            uint64_t s2[2] = {0ull, 0ull};
#pragma unroll
            for (int hb = 0; hb < CK / 64; ++hb) {
              const int k0 = (CK / 2) * h + 32 * hb;
              uint32_t pk[16];
#pragma unroll
              for (int i = 0; i < 32; i += 4) {
                float x[4];
                f32x2_unpack(f32x2_fma(f32x2_pack(v[k0 + i], v[k0 + i + 1]), sc2, nm2), x[0], x[1]);
                f32x2_unpack(f32x2_fma(f32x2_pack(v[k0 + i + 2], v[k0 + i + 3]), sc2, nm2), x[2], x[3]);
#pragma unroll
                for (int e = 0; e < 4; ++e) x[e] = ex2_approx(x[e]);
                uint64_t& acc = s2[(i >> 2) & 1];
                acc = f32x2_add(acc, f32x2_add(f32x2_pack(x[0], x[2]), f32x2_pack(x[1], x[3])));
                pk[i / 2] = pack_f16x2(x[0], x[1]);
                pk[i / 2 + 1] = pack_f16x2(x[2], x[3]);
              }
              tmem_st16_nowait(t_p + (uint32_t)(k0 / 2), pk);
            }
            float s0, s1, s3, s4;
            f32x2_unpack(s2[0], s0, s1);
            f32x2_unpack(s2[1], s3, s4);
            l[h] += (s0 + s1) + (s3 + s4);
          }
          tmem_st_wait();
          tc_fence_before();
          __syncwarp();
          mbar_arrive_if_at(bb + kSFull + 16u, go);
        }
        if (g > 0 && ++ps == NS) {
          ps = 0;
          ppar ^= 1u;
        }
      }
      // O / l of the unit as a split pair, once its last PV has completed
      // (chunk g - 1, at stage ps)
      if (active) {
        mbar_wait_at(bb + kKVE + 8u * (uint32_t)ps, ppar, p.status);
        tc_fence_after();
        // one plane (hi, lo) after the other through this warp's rows of the Q tile
        // (every S of the unit has read them; 16-byte pieces XOR-swizzled by
        // row: no bank conflicts), so that a store instruction writes whole row
        // pieces; a lane storing its own row touched 32 rows per instruction
        // (9000 cycles a unit with every group at it)
        float lt = l[0] + l[1];
        const int left = c.qcnt - c.q0 - (r & ~31);  // rows of this warp's block
        uint32_t hi[DH / 2], lo[DH / 2];
        {
          float o[DH];
          if constexpr (DH == 64)
            tmem_ld64(t_o, o);
          else
            tmem_ld32(t_o, o);
          if constexpr (SPLIT) {
            if (grp % p.ks != 0) {
#pragma unroll
              for (int k = 0; k < DH / 4; ++k)
                *reinterpret_cast<float4*>(part_row(grp, k)) =
                    make_float4(o[4 * k], o[4 * k + 1], o[4 * k + 2], o[4 * k + 3]);
              *part_ml(grp) = make_float2(m, lt);
            }
            set_sync();
            if (grp % p.ks == 0) {
              float mx = m;
              for (int g2 = grp + 1; g2 < grp + p.ks; ++g2) mx = fmaxf(mx, part_ml(g2)->x);
              float f = ex2_approx(m - mx);
              lt *= f;
#pragma unroll
              for (int i = 0; i < DH; ++i) o[i] *= f;
#pragma unroll 1
              for (int g2 = grp + 1; g2 < grp + p.ks; ++g2) {
                const float2 ml = *part_ml(g2);
                f = ex2_approx(ml.x - mx);
                lt = fmaf(ml.y, f, lt);
#pragma unroll
                for (int k = 0; k < DH / 4; ++k) {
                  const float4 x = *reinterpret_cast<const float4*>(part_row(g2, k));
                  o[4 * k] = fmaf(x.x, f, o[4 * k]);
                  o[4 * k + 1] = fmaf(x.y, f, o[4 * k + 1]);
                  o[4 * k + 2] = fmaf(x.z, f, o[4 * k + 2]);
                  o[4 * k + 3] = fmaf(x.w, f, o[4 * k + 3]);
                }
              }
            }
          }
          const float inv = 1.f / lt;
#pragma unroll
          for (int i = 0; i < DH / 2; ++i) split2(o[2 * i] * inv, o[2 * i + 1] * inv, hi[i], lo[i]);
        }
        const size_t blk = (size_t)(c.qoff + c.q0 + (r & ~31)) * p.ldo + p.o_col + head * DH;
        uint8_t* sOut = sQ + (u % NQ) * Cfg::kQBytes + q4 * Cfg::kQBlock;
        auto store = [&](bf16* dst, const uint32_t* w) {
#pragma unroll
          for (int k = 0; k < NC; ++k)
            *reinterpret_cast<uint4*>(sOut + lane * Cfg::kRowBytes + (((uint32_t)k ^ Cfg::swz(lane)) << 4)) =
                make_uint4(w[4 * k], w[4 * k + 1], w[4 * k + 2], w[4 * k + 3]);
          __syncwarp();
#pragma unroll
          for (int i = 0; i < NC; ++i) {
            const int row = (i * 32 + lane) / NC, ch = lane % NC;
            const uint4 v = *reinterpret_cast<const uint4*>(sOut + row * Cfg::kRowBytes + (((uint32_t)ch ^ Cfg::swz(row)) << 4));
            if (row < left && (!SPLIT || grp % p.ks == 0))
              *reinterpret_cast<uint4*>(dst + (size_t)row * p.ldo + ch * 8) = v;
          }
          __syncwarp();
        };
        store(p.o_h + blk, hi);
        store(p.o_l + blk, lo);
        tc_fence_before();  // read before the next unit's first PV overwrites it (p_full orders the two)
        fence_async_shared();  // staging read before the next load into these rows
        __syncwarp();
      } else if constexpr (SPLIT) {
        set_sync();
      }
      ++u;
    }
    // (after a timed-out wait, the Q rows still on their way)
    for (int v = u < NQ ? 0 : u - NQ; v < u; ++v)
      mbar_landed_at(bb + 8u * (uint32_t)(v % NQ), (uint32_t)(v / NQ) & 1u, p.status);
  }

  __syncwarp();
  tc_fence_before();
  __syncthreads();
  if (warp == 0) tmem_dealloc(*tmem_slot, 512);
}

namespace {
int g_attn_sms = 0;
constexpr int kSplitChunks = 32;  // of a unit, from which on groups share it
}

cudaError_t attn_prepare() {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&g_attn_sms, cudaDevAttrMultiProcessorCount, dev);
  auto smem = [&](const void* f, size_t n) {
    if (e == cudaSuccess) e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)n);
  };
  smem((const void*)attn_kernel<32, false>, AttnCfg<32>::kSmem);
  smem((const void*)attn_kernel<32, true>, AttnCfg<32>::kSmem);
  smem((const void*)attn_kernel<64, false>, AttnCfg<64>::kSmem);
  smem((const void*)attn_kernel<64, true>, AttnCfg<64>::kSmem);
  return e;
}

int attn_chunk_keys(int dh) { return dh == 32 ? AttnCfg<32>::CK : AttnCfg<64>::CK; }

cudaError_t attn_launch(int dh, const CUtensorMap* q, const CUtensorMap* k, const CUtensorMap* v, const AttnParams& p0,
                        cudaStream_t s) {
  if (p0.n_segments <= 0 || p0.max_q <= 0 || (!p0.kv_self && p0.kv_cnt <= 0)) return cudaSuccess;
  AttnParams p = p0;
  // the groups of a full grid take sb segments at a time, and with few of them several query tiles of each
  const int tiles = (p.max_q + BQ - 1) / BQ;
  const int sms = g_attn_sms > 0 ? g_attn_sms : 148;
  const int ng = dh == 32 ? AttnCfg<32>::NG : AttnCfg<64>::NG, groups = sms * ng;
  // Few units with many keys: as many groups as there are for each take a unit together
  // (SPLIT), from 32 chunks on.  Unsplit, a unit is one group's chain, 0.6 us a chunk and layer, and with
  // fewer units than groups the others stand idle: one request, d_h = 32, 2048 keys 134 us in all unsplit and
  // 109 split, 4096 179 and 128, 65536 1513 and 651; d_h = 64, 4096 keys 148 and 131; 16 requests of 16384 keys
  // 532 and 325; 64 requests of 4096 keys (two groups a unit) 247 split.  Below 32 chunks the order of the
  // sums stays the one group's.
  const int nch = (p.kv_cnt + attn_chunk_keys(dh) - 1) / attn_chunk_keys(dh);
  const long long units = (long long)p.n_segments * p.n_heads * tiles;
  p.ks = 1;
  if (!p.kv_self && nch >= kSplitChunks)
    for (p.ks = ng; p.ks > 1 && units * p.ks > groups;) p.ks /= 2;
  p.kper = (nch + p.ks - 1) / p.ks;
  if (p.ks > 1) {
    p.sb = p.n_segments;
    p.tp = tiles;
  } else {
    p.sb = groups / p.n_heads < p.n_segments ? groups / p.n_heads : p.n_segments;
    p.tp = groups / (p.sb * p.n_heads) < tiles ? groups / (p.sb * p.n_heads) : tiles;
  }
  const int w = p.sb * p.n_heads * p.tp;
  const dim3 g((unsigned)(w < sms ? w : sms));
  auto go = [&](auto kern, int threads, size_t smem) {
    return launch_k(kern, g, dim3((unsigned)threads), smem, s, *q, *k, *v, p);
  };
  if (dh == 32)
    return p.ks > 1 ? go(attn_kernel<32, true>, AttnCfg<32>::kThreads, AttnCfg<32>::kSmem)
                    : go(attn_kernel<32, false>, AttnCfg<32>::kThreads, AttnCfg<32>::kSmem);
  return p.ks > 1 ? go(attn_kernel<64, true>, AttnCfg<64>::kThreads, AttnCfg<64>::kSmem)
                  : go(attn_kernel<64, false>, AttnCfg<64>::kThreads, AttnCfg<64>::kSmem);
}

}  // namespace fe
