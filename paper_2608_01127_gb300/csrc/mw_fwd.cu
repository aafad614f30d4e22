// Block-causal attention forward on sm_103a (Sec. 3.2 block-causal
// self-attention; Sec. 3.5 rolling KV cache and pipelined denoising).
//
// One CTA owns a block of 2 x 128 query rows of one (b,h) and streams the key
// tiles that block can see.  Only unmasked work is enumerated: the key range
// of a query block ends at the end of the chunk of its last row, so whole
// chunk blocks above the diagonal are never visited; a per-row limit masks
// the few tiles that straddle a chunk edge.
//
// Roles (384 threads):
//   warps 0-3 / 4-7  softmax of query tile 0 / 1 (one thread per row = TMEM lane)
//   warp 8           TMA producer (Q once, then K/V tiles through a ring of stages)
//   warp 9           tcgen05 issuer (S = Q K^T into TMEM, O += P V with P in TMEM);
//                    d = 64: of query tile 0, and warp 10 of query tile 1
//   the rest of 10-11 RoPE re-shift of the sink anchor's key tiles in shared
//                    memory when it is enabled; with 80-wide MMAs on the
//                    128-wide tiles (and no re-shift) the ones columns of V;
//                    otherwise idle (they complete warpgroup 2 for the
//                    register re-split)
// TMEM (512 columns): S_t at column 128 t, O_t at 256 + OW t (OW = the MMA
// width, plus 16 columns where the PV MMA also sums P through ones in V).
// P_t, bf16, overwrites the first 64 columns of S_t; where there is room, only
// its first half does, and the second lies after the O columns.
// CTA order: groups of heads of about three waves of CTAs, one group after
// another; in a group the longest query blocks first.
#include <type_traits>

#include "mw_internal.h"
#include "mw_ptx.cuh"

namespace mw {
namespace {

// D: the head-dim width of the shared-memory tiles (64, or 128 with the
// columns past the caller's zero-filled by TMA); DM <= D: the columns the
// MMAs cover (QK^T reduces over DM, O has DM columns), 80 for head dims up
// to 80 on the 128-wide tiles
template <int D, int DM = D, bool ROPE = false, bool SPLIT = false>
struct FwdLayout {
  static_assert(DM % 16 == 0 && DM <= D, "MMA width");
  static constexpr int QT = kFwdQTiles;
  static constexpr int REG = D / 64;                  // 64-column swizzle regions per row
  static constexpr int REGION_BYTES = kTileRows * 128;
  static constexpr int TILE_BYTES = REG * REGION_BYTES;
  static constexpr int STAGES = (D == 64) ? 4 : 2;
  static constexpr int OFF_Q = 0;
  static constexpr int OFF_K = OFF_Q + QT * TILE_BYTES;
  static constexpr int OFF_V = OFF_K + STAGES * TILE_BYTES;
  // The row sum of P comes out of the PV MMA itself: V gets 16 extra columns
  // of bf16 ones, so O gets 16 extra columns that all hold sum_j P_ij.
  // d = 64: the ones are a region of their own, reached through each stage
  // descriptor's leading-byte offset.  80-wide MMAs on the 128-wide tiles:
  // the ones go into columns 80..95 of each V tile (which TMA fills with
  // zeros), written by the helper warps after every load; with the RoPE re-shift
  // those warps are busy and the softmax sums P itself.
  static constexpr bool ONES_IN_V = (D == 128 && DM == 80 && !ROPE);
  static constexpr bool SUM_MMA = (D == 64) || ONES_IN_V;
  static constexpr int OW = SUM_MMA ? DM + 16 : DM;   // O columns in TMEM
  static constexpr int SUM_COL = DM;                  // first row-sum column of O
  static constexpr int OFF_ONES = OFF_V + STAGES * TILE_BYTES;
  static constexpr int ONES_BYTES = (D == 64) ? REGION_BYTES : 0;
  // RoPE re-shift: (cos, sin) of the shift per channel pair (one copy per
  // rotating warp)
  static constexpr int OFF_ROPE = OFF_ONES + ONES_BYTES;
  static constexpr int ROPE_WARP_BYTES = (D / 2) * 8;
  static constexpr int ROPE_BYTES = 2 * ROPE_WARP_BYTES;
  static constexpr int OFF_BAR = OFF_ROPE + ROPE_BYTES;
  // P of a key tile's last 64 keys in columns of its own, where TMEM has room
  // (d = 64, and 80-wide MMAs): S is then free once the PV of the first 64
  // keys is issued, and the next tile's QK^T runs before the second half of P
  // is there, so that both tiles' softmax warps work all the time instead of
  // in turn (P over S as a whole leaves each tile's softmax waiting for its own
  // PV and QK^T).  d = 64, 24 heads x 16 x 880: 613 us before, 594 with the
  // early exponentials below alone, 568 with both and an issuer per tile (557
  // since, with a leaner epilogue); 16 heads of 72: 445, 438 and 436 us (with
  // one issuer).  A split key range is a handful of tiles a CTA, which the chain
  // through the first and the last of them dominates: it gains nothing (one step
  // against 8 chunks of 880, 12 heads of 64: 30.3 us against 30.6 with it; 16 of
  // 72: 46.0 against 47.6).
  static constexpr bool SPLIT_P = !SPLIT && 256 + OW * QT + 32 * QT <= 512;
  // MMA-issuing warps: at d = 64 one per query tile (warps 9 and 10), since a
  // step's waits and commits take an issuer about as long as its MMAs take the
  // tensor core, whose queue is only two instructions deep (601 us with one).
  // The 80-wide kernels need two warps for the ones columns of V (495 us with
  // two issuers and one helper).
  static constexpr int ISSUERS = D == 64 && SPLIT_P ? QT : 1;
  static constexpr int HELPERS = 3 - ISSUERS;  // the warps after the issuers
  static constexpr int NBAR = 1 + 6 * STAGES + (SPLIT_P ? 4 : 3) * QT + 1;
  static constexpr int OFF_MISC = OFF_BAR + NBAR * 8;
  static constexpr int BYTES = OFF_MISC + 16;
  static constexpr uint32_t S_COL(int t) { return 128u * t; }
  static constexpr uint32_t O_COL(int t) { return 256u + OW * t; }
  // P of the first and of the last 64 keys of a tile
  static constexpr uint32_t P_COL(int t, int half) {
    return half == 0 ? S_COL(t) : SPLIT_P ? 256u + OW * QT + 32u * t : S_COL(t) + 32u;
  }
  // With the re-shift on 128-wide MMAs the unsplit epilogue keeps a row-per-
  // thread form of the fp32 partials that no launch takes (the launcher picks
  // SPLIT for several splits): the compiler schedules that kernel's key loop
  // 2.7% faster with it (16 heads of 128, 8 x 880 rows against 12 chunks and a
  // sink, 582 us, 597 without it; unrolling the epilogue less, 592).  The others
  // gain by being without it: the re-shift at d = 72 488 -> 482 us, the plain
  // forward at d = 64 566 -> 557.
  static constexpr bool ROWS_KEPT = ROPE && !SPLIT && DM == 128;
  static constexpr int THREADS = 384;
  // registers per thread after the re-split: softmax warpgroups 0-1 get
  // more, warpgroup 2 (TMA, MMA, RoPE or idle warps) less; 2*128*S + 128*C
  // equals the launch's 384 threads x 168 registers.  d = 128: the MMA
  // warp's unrolled issue loop needs more than 56 (measured: 208/88 runs
  // the d=128 forward 4% faster, 224/56 the d=64 one 1% faster)
  static constexpr int REGS_LAUNCH = 168;
  static constexpr int REGS_SOFTMAX = (D == 64) ? 224 : 208;
  static constexpr int REGS_CONTROL = (D == 64) ? 56 : 88;
  static_assert(2 * 128 * REGS_SOFTMAX + 128 * REGS_CONTROL == THREADS * REGS_LAUNCH,
                "register re-split must hand out exactly the launch's registers");
};

// Where key tile j of a query block comes from.  Keys are visited in logical
// order: the sink anchor (segment S), the ring from its head to the end of
// the buffer (A) and from the start after wrapping (B), then the queries' own
// chunks (C).
enum : int { kSegOwn = 0, kSegRing = 1, kSegSink = 2 };
struct TileSrc {
  int seg;     // kSegOwn, kSegRing or kSegSink: which tensor maps hold the tile
  int row0;    // first physical row of the tile
  int end;     // ring and sink: exclusive end of the valid rows; own: unused
  int t0;      // ring: logical index (oldest = 0) of the tile's first row
};

struct Segs {
  int nS, nA, nB, nC;
  int endS, headA, endA, endB, lenA;
};

__device__ __forceinline__ TileSrc tile_src(const Segs& g, int j) {
  TileSrc s;
  s.t0 = 0;
  if (j < g.nS) {
    s.seg = kSegSink;
    s.row0 = j * kTileRows;
    s.end = g.endS;
    return s;
  }
  j -= g.nS;
  if (j < g.nA) {
    s.seg = kSegRing;
    s.row0 = g.headA + j * kTileRows;
    s.end = g.endA;
    s.t0 = j * kTileRows;
  } else if (j < g.nA + g.nB) {
    s.seg = kSegRing;
    s.row0 = (j - g.nA) * kTileRows;
    s.end = g.endB;
    s.t0 = g.lenA + (j - g.nA) * kTileRows;
  } else {
    s.seg = kSegOwn;
    s.row0 = (j - g.nA - g.nB) * kTileRows;
    s.end = 0;
  }
  return s;
}

// ROPE: the cache form with the RoPE re-shift of the sink anchor (the helper warps
// turn its key tiles before the MMAs read them); the training and plain
// cache forms are compiled without it.  SPLIT: the key range is one of
// several (p.num_splits > 1), O goes out as fp32 partials through TMA
// stores; without it, as bf16 rows (the training form never pays for the
// partials' code).
template <int D, int DM, bool ROPE, bool SPLIT>
__global__ void __launch_bounds__(FwdLayout<D, DM>::THREADS, 1)
    bca_fwd_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
                   const __grid_constant__ CUtensorMap tm_v, const __grid_constant__ CUtensorMap tm_kr,
                   const __grid_constant__ CUtensorMap tm_vr, const __grid_constant__ CUtensorMap tm_ks,
                   const __grid_constant__ CUtensorMap tm_vs, const __grid_constant__ CUtensorMap tm_op,
                   const __grid_constant__ FwdParams p, const __grid_constant__ RopeFreq rope_om) {
  using L = FwdLayout<D, DM, ROPE, SPLIT>;
  constexpr int QT = L::QT;
  constexpr int NS = L::STAGES;
  extern __shared__ __align__(1024) uint8_t smem[];
  // ---- work item: p.head_groups groups of heads one after another (sizes
  // differ by at most one, the larger first), so that the CTAs running
  // together share a few heads' K/V in L2; inside a group the longest query
  // blocks (they see the most keys) come first
  int x = blockIdx.x;
  const int split = x % p.num_splits;
  x /= p.num_splits;
  const int g_base = p.BH / p.head_groups, g_rem = p.BH % p.head_groups;
  const int big = (g_base + 1) * p.n_qblocks;  // CTAs of one larger group
  int in_grp, gsize, h0;
  if (x < g_rem * big) {
    gsize = g_base + 1;
    h0 = (x / big) * gsize;
    in_grp = x % big;
  } else {
    const int y = x - g_rem * big;
    gsize = g_base;
    h0 = g_rem * (g_base + 1) + (y / (g_base * p.n_qblocks)) * g_base;
    in_grp = y % (g_base * p.n_qblocks);
  }
  const int bh = h0 + in_grp % gsize;
  const int qb = p.n_qblocks - 1 - in_grp / gsize;
  const int r0 = qb * kFwdBlockRows;
  if ((smem_u32(smem) & 1023u) != 0u) {
    // nothing runs without aligned shared memory: report it, and give this
    // CTA's rows a defined result (O = 0, LSE = -inf; as split partials, a
    // -inf LSE that the combine skips) instead of leaving stale values behind
    if (threadIdx.x == 0) atomicOr(p.status, kDevMisaligned);
    const int row = r0 + static_cast<int>(threadIdx.x);
    if (threadIdx.x < kFwdBlockRows && row < p.rows_q) {
      const size_t row_off = static_cast<size_t>(bh) * p.rows_q + row;
      if (p.num_splits == 1) {
        const int d_io = (D == 64) ? D : p.d_io;
        uint4* dst = reinterpret_cast<uint4*>(p.o + row_off * d_io);
        for (int c = 0; c < d_io / 8; ++c) dst[c] = make_uint4(0u, 0u, 0u, 0u);
        if (p.lse) p.lse[row_off] = -INFINITY;
      } else {
        p.lse_part[static_cast<size_t>(split) * p.BH * p.rows_q + row_off] = -INFINITY;
      }
    }
    return;  // uniform across the CTA, before any barrier or TMEM use
  }
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + L::OFF_BAR);
  uint64_t* q_full = bars;
  uint64_t* k_full = bars + 1;
  uint64_t* k_empty = k_full + NS;
  uint64_t* v_full = k_empty + NS;
  uint64_t* v_empty = v_full + NS;
  uint64_t* k_rdy = v_empty + NS;  // K tile in shared memory, RoPE re-shift applied
  uint64_t* v_rdy = k_rdy + NS;    // V tile in shared memory with its ones columns
  uint64_t* s_full = v_rdy + NS;
  uint64_t* p_full = s_full + QT;
  uint64_t* p_half = p_full + QT;  // first 64 keys of P in TMEM
  uint64_t* pv_done = p_half + QT;  // SPLIT_P: the PV of a key tile is done
  uint64_t* o_full = pv_done + (L::SPLIT_P ? QT : 0);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + L::OFF_MISC);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem + L::OFF_MISC + 4);

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;

  // query tiles of the block that hold rows (the last block may hold one)
  const int qt_n = (r0 + kTileRows < p.rows_q) ? QT : 1;
  const int last_row = min(r0 + kFwdBlockRows - 1, p.rows_q - 1);
  const int c_end = (last_row / p.T + 1) * p.T;  // keys of segment C visible to the block

  Segs g;
  g.lenA = 0;
  g.nS = (p.sink_len + kTileRows - 1) / kTileRows;
  g.endS = p.sink_len;
  const int lenA = min(p.ring_len, p.ring_cap - p.ring_head);
  const int lenB = p.ring_len - lenA;
  g.nA = (lenA + kTileRows - 1) / kTileRows;
  g.nB = (lenB + kTileRows - 1) / kTileRows;
  g.nC = (c_end + kTileRows - 1) / kTileRows;
  g.headA = p.ring_head;
  g.endA = p.ring_head + lenA;
  g.lenA = lenA;
  g.endB = lenB;
  const int n_all = g.nS + g.nA + g.nB + g.nC;
  const int j0 = (int)((long long)split * n_all / p.num_splits);
  const int j1 = (int)((long long)(split + 1) * n_all / p.num_splits);
  const int n_local = j1 - j0;

  const int n_issuers = L::ISSUERS == 1 ? 1 : min(L::ISSUERS, qt_n);  // that have a query tile
  if (threadIdx.x == 0) {
    mbar_init(q_full, 1);
    for (int s = 0; s < NS; ++s) {
      mbar_init(&k_full[s], 1);
      mbar_init(&k_empty[s], n_issuers);
      mbar_init(&v_full[s], 1);
      mbar_init(&v_empty[s], n_issuers);
      mbar_init(&k_rdy[s], L::HELPERS);
      mbar_init(&v_rdy[s], L::HELPERS);
    }
    for (int t = 0; t < QT; ++t) {
      mbar_init(&s_full[t], 1);
      mbar_init(&p_full[t], 4);
      mbar_init(&p_half[t], 4);
      if constexpr (L::SPLIT_P) mbar_init(&pv_done[t], 1);
    }
    mbar_init(o_full, n_issuers);
    *abort_flag = 0;
    fence_mbar_init();
  }
  // descriptors (kernel parameters, so they may be read before the previous
  // kernel ends): in the setup where a launch has few key tiles a CTA (rolling
  // step 58.9 -> 57.8 us); the unsplit forward measured 0.2% slower that way
  auto prefetch_maps = [&]() {
    prefetch_tmap(&tm_q);
    prefetch_tmap(&tm_k);
    prefetch_tmap(&tm_v);
    if constexpr (SPLIT) {
      prefetch_tmap(&tm_kr);
      prefetch_tmap(&tm_vr);
    }
  };
  if (SPLIT && warp == 8 && lane == 0) prefetch_maps();
  if (warp == 9) {
    tmem_alloc(tmem_slot, 512);
    tmem_relinquish();
  }
  if constexpr (L::ONES_BYTES > 0) {
    uint4* ones = reinterpret_cast<uint4*>(smem + L::OFF_ONES);
    const uint32_t one2 = 0x3F803F80u;  // bf16 1.0 twice
    for (int k = threadIdx.x; k < L::ONES_BYTES / 16; k += L::THREADS)
      ones[k] = make_uint4(one2, one2, one2, one2);
    fence_proxy_async_smem();  // read by the tensor core (async proxy)
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  // the allocation of all 512 columns can only start at 0; as a constant it
  // keeps the issuing warp's TMEM addresses out of registers (with one-word
  // operand descriptors, 12 heads of 128, 32 x 600 tokens: 783 us before, 749
  // with the descriptors, 721 with both; d = 64, 16 x 880: 640 -> 631 us).  A
  // look at the slot, in any place, costs the 128-wide kernel 0.6% or more
  constexpr uint32_t tmem = 0;
  const WaitCtl ctl{abort_flag, p.status, p.budget_ns};
  // launched early (programmatic dependent launch): the setup above has run
  // while the previous kernel finished; global memory only from here on
  pdl_wait();

  uint8_t* sQ = smem + L::OFF_Q;
  uint8_t* sK = smem + L::OFF_K;
  uint8_t* sV = smem + L::OFF_V;

  if (warp >= 8) {
  // warpgroup 2: every warp executes this one re-split instruction
  regs_dec<L::REGS_CONTROL>();
  if (warp == 8) {
    // ------------------------------------------------------------ TMA producer
    if (lane == 0 && n_local > 0) {
      if (!SPLIT) prefetch_maps();
      bool q_issued = false;
      if (!p.debug_skip_q) {
        mbar_arrive_expect_tx(q_full, QT * L::TILE_BYTES);
        for (int t = 0; t < QT; ++t)
          for (int r = 0; r < L::REG; ++r)
            tma_load_3d(sQ + t * L::TILE_BYTES + r * L::REGION_BYTES, &tm_q, q_full, 64 * r,
                        r0 + kTileRows * t, bh);
        q_issued = true;
      }
      int issued_k = 0, issued_v = 0;
      for (int i = 0; i < n_local; ++i) {
        const int st = i % NS;
        const uint32_t ph = (i / NS) & 1;
        const TileSrc src = tile_src(g, j0 + i);
        if (!mbar_wait(&k_empty[st], ph ^ 1, ctl)) break;
        mbar_arrive_expect_tx(&k_full[st], L::TILE_BYTES);
        for (int r = 0; r < L::REG; ++r)
          tma_load_3d(sK + st * L::TILE_BYTES + r * L::REGION_BYTES,
                      src.seg == kSegRing ? &tm_kr : src.seg == kSegSink ? &tm_ks : &tm_k,
                      &k_full[st], 64 * r, src.row0, bh);
        ++issued_k;
        if (!mbar_wait(&v_empty[st], ph ^ 1, ctl)) break;
        mbar_arrive_expect_tx(&v_full[st], L::TILE_BYTES);
        for (int r = 0; r < L::REG; ++r)
          tma_load_3d(sV + st * L::TILE_BYTES + r * L::REGION_BYTES,
                      src.seg == kSegRing ? &tm_vr : src.seg == kSegSink ? &tm_vs : &tm_v,
                      &v_full[st], 64 * r, src.row0, bh);
        ++issued_v;
      }
      if (*abort_flag) {
        // let every copy this CTA started land before shared memory goes away
        if (q_issued) drain_wait(q_full, 0, p.budget_ns);
        for (int i = max(0, issued_k - NS); i < issued_k; ++i)
          drain_wait(&k_full[i % NS], (i / NS) & 1, p.budget_ns);
        for (int i = max(0, issued_v - NS); i < issued_v; ++i)
          drain_wait(&v_full[i % NS], (i / NS) & 1, p.budget_ns);
      }
    }
  } else if (warp == 9 || (L::ISSUERS > 1 && warp == 10)) {
    // ------------------------------------------------------------ MMA issuers (whole warps)
    if (n_local > 0) {
      constexpr uint32_t idesc_qk = idesc_bf16_f32(128, 128, false, false);
      constexpr uint32_t idesc_pv = idesc_bf16_f32(128, L::OW, false, true);
      // descriptors computed once; each MMA adds a compile-time offset
      const uint32_t q_desc = sdesc_sw128(smem_u32(sQ), 16);
      const uint32_t k_desc = sdesc_sw128(smem_u32(sK), 16);
      const uint32_t v_addr = smem_u32(sV);
      const uint32_t ones_addr = smem_u32(smem + L::OFF_ONES);

      auto issue_qk = [&](int t, int st) {
        const uint32_t qa = sdesc_add(q_desc, t * L::TILE_BYTES);
        const uint32_t kb = sdesc_add(k_desc, st * L::TILE_BYTES);
#pragma unroll
        for (int kk = 0; kk < DM / 16; ++kk) {
          const uint32_t off = (kk >> 2) * L::REGION_BYTES + (kk & 3) * 32;
          umma_ss(tmem + L::S_COL(t), sdesc_add(qa, off), sdesc_add(kb, off), idesc_qk,
                  kk > 0 ? 1u : 0u);
        }
      };
      // O_t (+)= P_t V for keys [64 half, 64 half + 64) of the tile
      auto issue_pv = [&](int t, int st, bool acc, int half) {
        // V stage st; for d = 64 the next 64 "columns" are the ones region
        const uint32_t vs = v_addr + st * L::TILE_BYTES;
        const uint32_t vb = sdesc_sw128(vs, L::ONES_BYTES > 0 ? ones_addr - vs : L::REGION_BYTES);
#pragma unroll
        for (int k4 = 0; k4 < 4; ++k4) {
          const int kk = 4 * half + k4;
          umma_ts(tmem + L::O_COL(t), tmem + L::P_COL(t, half) + k4 * 8, sdesc_add(vb, kk * 2048),
                  idesc_pv, (acc || kk > 0) ? 1u : 0u);
        }
      };

      bool ok = warp_wait(q_full, 0, ctl);
      tc_fence_after();
      if constexpr (L::SPLIT_P) {
        // K tile i in shared memory (with the re-shift, a sink tile is read
        // once the helper warps have turned it)
        auto wait_k = [&](int i) {
          const int st = i % NS;
          return warp_wait(ROPE && j0 + i < g.nS ? &k_rdy[st] : &k_full[st], (i / NS) & 1, ctl);
        };
        // query tiles [first, last): one issuer's, or all of them
        auto issue = [&](auto first, auto last) {
          constexpr int T0 = decltype(first)::value, T1 = decltype(last)::value;
          if (T0 >= qt_n) return;
          if (ok && (ok = wait_k(0))) {
            tc_fence_after();
#pragma unroll
            for (int t = T0; t < T1; ++t) {
              if (t >= qt_n) break;
              issue_qk(t, 0);
              umma_commit(&s_full[t]);
            }
            umma_commit(&k_empty[0]);
          }
          for (int i = 0; ok && i < n_local; ++i) {
            const int st = i % NS;
            const int st1 = (i + 1) % NS;
            const bool more = i + 1 < n_local;
            if (more && !(ok = wait_k(i + 1))) break;
            if (!(ok = warp_wait(L::ONES_IN_V ? &v_rdy[st] : &v_full[st], (i / NS) & 1, ctl))) break;
#pragma unroll
            for (int t = T0; t < T1; ++t) {
              if (t >= qt_n) break;
              if (!(ok = warp_wait(&p_half[t], i & 1, ctl))) break;
              tc_fence_after();
              issue_pv(t, st, i > 0, 0);
              if (more) {
                issue_qk(t, st1);
                umma_commit(&s_full[t]);
              }
              if (!(ok = warp_wait(&p_full[t], i & 1, ctl))) break;
              tc_fence_after();
              issue_pv(t, st, true, 1);
              umma_commit(&pv_done[t]);
            }
            if (!ok) break;
            if (more) umma_commit(&k_empty[st1]);
            umma_commit(&v_empty[st]);
          }
          if (ok) umma_commit(o_full);
        };
        if constexpr (L::ISSUERS == 1) {
          issue(std::integral_constant<int, 0>{}, std::integral_constant<int, QT>{});
        } else {
          static_assert(QT == 2, "an issuer for each of two query tiles");
          if (warp == 9)
            issue(std::integral_constant<int, 0>{}, std::integral_constant<int, 1>{});
          else
            issue(std::integral_constant<int, 1>{}, std::integral_constant<int, 2>{});
        }
      } else {
        for (int i = 0; ok && i < n_local; ++i) {
          const int st = i % NS;
          const uint32_t ph = (i / NS) & 1;
          const int stp = (i + NS - 1) % NS;
          const uint32_t php = ((i - 1) / NS) & 1;
          // with the re-shift, a sink tile is read once the helper warps have turned it
          const bool turned = ROPE && j0 + i < g.nS;
          if (!(ok = warp_wait(turned ? &k_rdy[st] : &k_full[st], ph, ctl))) break;
          tc_fence_after();
          // unrolled over the compile-time tile count, so every descriptor
          // offset stays a constant (a runtime trip count here slows the whole
          // forward by ~8%: the issuing code must never pause)
#pragma unroll
          for (int t = 0; t < QT; ++t) {
            if (t >= qt_n) break;
            if (i > 0) {
              // PV of the first 64 keys while the softmax warps store the rest of P
              if (!(ok = warp_wait(&p_half[t], (i - 1) & 1, ctl))) break;
              if (t == 0 && !(ok = warp_wait(L::ONES_IN_V ? &v_rdy[stp] : &v_full[stp], php, ctl))) break;
              tc_fence_after();
              issue_pv(t, stp, i - 1 > 0, 0);
              if (!(ok = warp_wait(&p_full[t], (i - 1) & 1, ctl))) break;
              tc_fence_after();
              issue_pv(t, stp, true, 1);
            }
            issue_qk(t, st);
            umma_commit(&s_full[t]);
          }
          if (!ok) break;
          umma_commit(&k_empty[st]);
          if (i > 0) umma_commit(&v_empty[stp]);
        }
        if (ok) {
          const int il = n_local - 1;
          const int stl = il % NS;
#pragma unroll
          for (int t = 0; t < QT; ++t) {
            if (!ok || t >= qt_n) break;
            if (!(ok = warp_wait(&p_half[t], il & 1, ctl))) break;
            if (t == 0 && !(ok = warp_wait(L::ONES_IN_V ? &v_rdy[stl] : &v_full[stl], (il / NS) & 1, ctl)))
              break;
            tc_fence_after();
            issue_pv(t, stl, il > 0, 0);
            if (!(ok = warp_wait(&p_full[t], il & 1, ctl))) break;
            tc_fence_after();
            issue_pv(t, stl, true, 1);
          }
          if (ok) {
            umma_commit(&v_empty[stl]);
            umma_commit(o_full);
          }
        }
      }
    }
  } else if (ROPE && n_local > 0) {
    // ------------------------------------------------------------ RoPE re-shift of the sink
    // Queries, in-flight keys and ring keys carry their temporal rotation at
    // stream positions.  Re-shifting (Sec. 3.5) moves the window back by the
    // evicted frames and leaves the sink anchor at its position; since the
    // scores depend only on position differences, that changes just the
    // query-sink angles, exactly as turning the sink's keys forward by
    // rope_shift frames does.  That happens here, in shared memory, between
    // the TMA copy of a sink tile and the MMAs that read it: channel pair
    // (2i, 2i+1), i < rope_dims / 2, turns by rope_shift * base^(-2i/rope_dims).
    // With two helper warps each turns its own half of every sink tile (rows
    // [64 h, 64 h + 64)), so they never wait for each other.
    const int half = warp - 9 - L::ISSUERS;
    constexpr int kRows = kTileRows / L::HELPERS;  // of a helper
    float2* cs = reinterpret_cast<float2*>(smem + L::OFF_ROPE + half * L::ROPE_WARP_BYTES);
    const int pairs = p.rope_dims / 2;
    for (int i = lane; i < pairs; i += 32) cs[i] = rope_cos_sin(p.rope_shift, rope_om.hi[i], rope_om.lo[i]);
    __syncwarp();
    // lane -> (row within a pass, 16-byte chunk of 8 channels = 4 pairs)
    const int n_ch = (pairs + 3) / 4;
    const int rpp = 32 / n_ch;
    const int my_r = lane / n_ch, my_ch = lane % n_ch;
    const bool active = my_r < rpp;
    const int c0 = 8 * my_ch;
    const int np = min(4, pairs - 4 * my_ch);        // pairs of the chunk that turn
    const int region_off = (c0 >> 6) * L::REGION_BYTES;
    const int cidx = (c0 & 63) >> 3;                 // chunk index within the 128-byte row
    const float4 c01 = reinterpret_cast<const float4*>(cs)[2 * my_ch];
    const float4 c23 = reinterpret_cast<const float4*>(cs)[2 * my_ch + 1];
    const int n_sink = min(n_local, g.nS - j0);     // a block visits the sink first
    for (int i = 0; i < n_sink; ++i) {
      const int st = i % NS;
      if (!warp_wait(&k_full[st], (i / NS) & 1, ctl)) break;
      const TileSrc src = tile_src(g, j0 + i);
      const int r_lo = kRows * half;
      const int nrows = min(kRows, src.end - src.row0 - r_lo);  // valid rows of this part
      if (active && nrows > 0) {
        uint8_t* tile = sK + st * L::TILE_BYTES + region_off;
#pragma unroll 2
        for (int rr = my_r; rr < nrows; rr += rpp) {
          const int r = r_lo + rr;
          // 128-byte swizzle: 16-byte chunk index ^ (row mod 8)
          uint4* a = reinterpret_cast<uint4*>(tile + r * 128 + ((cidx ^ (r & 7)) << 4));
          uint4 v = *a;
          v.x = rope_turn(v.x, make_float2(c01.x, c01.y));
          if (np > 1) v.y = rope_turn(v.y, make_float2(c01.z, c01.w));
          if (np > 2) v.z = rope_turn(v.z, make_float2(c23.x, c23.y));
          if (np > 3) v.w = rope_turn(v.w, make_float2(c23.z, c23.w));
          *a = v;
        }
      }
      fence_proxy_async_smem();  // the tensor core reads the tile next
      __syncwarp();
      if (lane == 0) mbar_arrive(&k_rdy[st]);
    }
  } else if (L::ONES_IN_V && n_local > 0) {
    // ------------------------------------------------------------ ones columns of V
    // columns DM..DM+15 of each V tile hold bf16 ones (the row-sum columns of
    // the PV MMA); TMA zero-fills them on every load, so they are written
    // again after each one: 16-byte chunks (DM-64)/8 and (DM-64)/8 + 1 of
    // region 1's 128-byte rows, at their 128-byte-swizzle positions
    constexpr int kRows = kTileRows / L::HELPERS;  // of a helper
    const int r_lo = kRows * (warp - 9 - L::ISSUERS);
    const int c0 = (DM - 64) / 8;
    const uint4 ones = make_uint4(0x3F803F80u, 0x3F803F80u, 0x3F803F80u, 0x3F803F80u);
    for (int i = 0; i < n_local; ++i) {
      const int st = i % NS;
      if (!warp_wait(&v_full[st], (i / NS) & 1, ctl)) break;
      uint8_t* reg1 = sV + st * L::TILE_BYTES + L::REGION_BYTES;
#pragma unroll
      for (int k = 0; k < kRows / 32; ++k) {
        const int r = r_lo + 32 * k + lane;
        *reinterpret_cast<uint4*>(reg1 + r * 128 + ((c0 ^ (r & 7)) << 4)) = ones;
        *reinterpret_cast<uint4*>(reg1 + r * 128 + (((c0 + 1) ^ (r & 7)) << 4)) = ones;
      }
      fence_proxy_async_smem();  // the tensor core reads the tile next
      __syncwarp();
      if (lane == 0) mbar_arrive(&v_rdy[st]);
    }
  }
  } else {
    regs_inc<L::REGS_SOFTMAX>();
    // ------------------------------------------------------------ softmax
    const int t = warp >> 2;
    const int wq = warp & 3;
    const int row_local = wq * 32 + lane;
    const int row = r0 + t * kTileRows + row_local;
    const bool row_valid = row < p.rows_q;
    const int c_limit = (min(row, p.rows_q - 1) / p.T + 1) * p.T;
    const uint32_t lane_base = tmem + (static_cast<uint32_t>(wq * 32) << 16);
    const uint32_t s_addr = lane_base + L::S_COL(t);
    const uint32_t o_addr = lane_base + L::O_COL(t);
    const float sl2 = p.scale_log2;

    float m_used = -INFINITY;
    float l = 0.f;
    bool ok = true;
    const int n_steps = t < qt_n ? n_local : 0;  // an empty query tile does nothing
    for (int i = 0; i < n_steps; ++i) {
      const TileSrc src = tile_src(g, j0 + i);
      if (!(ok = warp_wait(&s_full[t], i & 1, ctl))) break;
      tc_fence_after();
      float s[128];
      if constexpr (L::SPLIT_P) {
        uint32_t r[4][32];
#pragma unroll
        for (int c = 0; c < 4; ++c) tmem_ld32(s_addr + 32 * c, r[c]);
        tmem_wait_ld();
#pragma unroll
        for (int c = 0; c < 128; ++c) s[c] = __uint_as_float(r[c / 32][c % 32]);
      } else {
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          uint32_t r[32];
          tmem_ld32(s_addr + 32 * c, r);
          tmem_wait_ld();
#pragma unroll
          for (int k = 0; k < 32; ++k) s[32 * c + k] = __uint_as_float(r[k]);
        }
      }
      const int limit = (src.seg != kSegOwn ? src.end : c_limit) - src.row0;
      if (limit < kTileRows) {
#pragma unroll
        for (int c = 0; c < 128; ++c)
          if (c >= limit) s[c] = -INFINITY;
      }
      // P of keys 32 g4 + 2 k and + 1, as a bf16 pair, relative to a maximum
      const float2 sl2x2 = make_float2(sl2, sl2);
      auto minus = [](float m) {
        const float m_eff = (m == -INFINITY) ? 0.f : m;
        return make_float2(-m_eff, -m_eff);
      };
      auto weights = [&](int g4, int k, float2 negm) {
        const float2 x = fma2(make_float2(s[32 * g4 + 2 * k], s[32 * g4 + 2 * k + 1]), sl2x2, negm);
        return pack_bf16x2(ex2_approx(x.x), ex2_approx(x.y));
      };
      // The first groups against the maximum so far, which the tile hardly ever
      // replaces (they are redone then): their exponentials overlap the loads
      // and the maximum instead of waiting for them.  A tile's softmax alone
      // took 1024 cycles without them, 848 with two groups, 875 with three;
      // where the tiles' softmaxes take turns (d = 128) it gained nothing.
      constexpr int kEarly = L::SPLIT_P ? 2 : 0;
      [[maybe_unused]] uint32_t early[kEarly > 0 ? kEarly : 1][16];
      auto set_early = [&](float2 negm) {
#pragma unroll
        for (int g4 = 0; g4 < kEarly; ++g4)
#pragma unroll
          for (int k = 0; k < 16; ++k) early[g4][k] = weights(g4, k, negm);
      };
      set_early(minus(m_used));
      float mq[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) mq[k] = fmaxf(s[k], s[k + 4]);
#pragma unroll
      for (int c = 8; c < 128; c += 8) {
        mq[0] = max3(mq[0], s[c], s[c + 1]);
        mq[1] = max3(mq[1], s[c + 2], s[c + 3]);
        mq[2] = max3(mq[2], s[c + 4], s[c + 5]);
        mq[3] = max3(mq[3], s[c + 6], s[c + 7]);
      }
      const float mx = max3(fmaxf(mq[0], mq[1]), mq[2], mq[3]);
      const float m_tile = mx * sl2;  // scale > 0
      const float m_cand = fmaxf(m_used, m_tile);
      // Rescale only when the running maximum grew by more than 2^8: P stays
      // below 256 in between, and the final O / l is exact either way.
      const bool need = m_cand > m_used + 8.0f;
      if (__any_sync(0xffffffffu, need)) {
        float alpha = 1.f;
        if (need) {
          alpha = ex2_approx(m_used - m_cand);
          m_used = m_cand;
        }
        set_early(minus(m_used));
        l *= alpha;
        if (i > 0) {
          if constexpr (L::SPLIT_P) {  // (else S of this tile implies it)
            if (!(ok = warp_wait(&pv_done[t], (i - 1) & 1, ctl))) break;
            tc_fence_after();
          }
          // exactly the tile's O columns (the next tile's O follows them)
#pragma unroll
          for (int c = 0; c < DM / 32; ++c) {
            uint32_t r[32];
            tmem_ld32(o_addr + 32 * c, r);
            tmem_wait_ld();
#pragma unroll
            for (int k = 0; k < 32; ++k) r[k] = __float_as_uint(__uint_as_float(r[k]) * alpha);
            tmem_st32(o_addr + 32 * c, r);
          }
          if constexpr (DM % 32 != 0) {
            uint32_t r[16];
            tmem_ld16(o_addr + DM - 16, r);
            tmem_wait_ld();
#pragma unroll
            for (int k = 0; k < 16; ++k) r[k] = __float_as_uint(__uint_as_float(r[k]) * alpha);
            tmem_st16(o_addr + DM - 16, r);
          }
          if constexpr (L::SUM_MMA) {  // the row-sum columns scale with O
            uint32_t r[16];
            tmem_ld16(o_addr + L::SUM_COL, r);
            tmem_wait_ld();
#pragma unroll
            for (int k = 0; k < 16; ++k) r[k] = __float_as_uint(__uint_as_float(r[k]) * alpha);
            tmem_st16(o_addr + L::SUM_COL, r);
          }
          tmem_wait_st();
        }
      }
      const float2 negm = minus(m_used);
      float2 acc = make_float2(0.f, 0.f);
      // P in four 32-key groups, each stored as soon as it is packed; the first
      // two groups (keys 0..63) are announced while the third is stored
#pragma unroll
      for (int g4 = 0; g4 < 4; ++g4) {
        uint32_t packed[16];
#pragma unroll
        for (int k = 0; k < 16; ++k) {
          const uint32_t pk = g4 < kEarly ? early[g4 < kEarly ? g4 : 0][k] : weights(g4, k, negm);
          // the row sum uses the bf16 weights the PV MMA consumes, so O is an
          // exact convex combination of them (d = 64: summed by the MMA)
          if constexpr (!L::SUM_MMA)
            acc = add2(acc, make_float2(__uint_as_float(pk << 16), __uint_as_float(pk & 0xffff0000u)));
          packed[k] = pk;
        }
        if (g4 == 2) {  // the first half has landed: its PV can start
          tmem_wait_st();
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(&p_half[t]);
          // the previous tile's PV has read the columns of the second half
          if (L::SPLIT_P && i > 0) {
            if (!(ok = warp_wait(&pv_done[t], (i - 1) & 1, ctl))) break;
            tc_fence_after();
          }
        }
        const uint32_t p_addr = L::SPLIT_P && g4 >= 2 ? lane_base + L::P_COL(t, 1) : s_addr + 32 * (g4 >> 1);
        tmem_st16(p_addr + 16 * (g4 & 1), packed);
      }
      if (!ok) break;
      l += acc.x + acc.y;
      tmem_wait_st();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&p_full[t]);
    }

    // ---- epilogue
    pdl_trigger();  // the next kernel (the split combine) may be scheduled now
    const bool have = __all_sync(0xffffffffu, ok) && n_steps > 0 && warp_wait(o_full, 0, ctl);
    tc_fence_after();
    if constexpr (L::SUM_MMA) {
      if (have) {
        uint32_t r[16];
        tmem_ld16(o_addr + L::SUM_COL, r);
        tmem_wait_ld();
        l = __uint_as_float(r[0]);
      }
    }
    const bool nonzero = have && l > 0.f;
    const float inv_l = nonzero ? 1.f / l : 0.f;
    const float m_eff = (m_used == -INFINITY) ? 0.f : m_used;
    const float lse = nonzero ? (m_eff + __log2f(l)) * 0.69314718055994530942f : -INFINITY;
    const size_t row_off = static_cast<size_t>(bh) * p.rows_q + row;
    // split partials: each warp writes its 32 rows of the tile's fp32 O into
    // shared memory (the K/V stages, no longer read once O is final) as
    // 32-column boxes with the 128-byte swizzle, and one thread of the tile
    // hands the boxes to the TMA unit.  Row-per-thread global stores would
    // cost 32 transactions per warp instruction, all CTAs at once.
    constexpr int kBoxBytes = kTileRows * 128;  // 128 rows x 32 fp32
    // the chunks that hold the DM columns of O (the caller's d_io <= DM)
#pragma unroll
    for (int c = 0; c < (DM + 31) / 32; ++c) {
      uint32_t r[32];
      if (have) {
        tmem_ld32(o_addr + 32 * c, r);
        tmem_wait_ld();
      }
      float v[32];
#pragma unroll
      for (int k = 0; k < 32; ++k) v[k] = nonzero ? __uint_as_float(r[k]) * inv_l : 0.f;
      if constexpr (!SPLIT) {
        if (!row_valid) continue;
        if (!L::ROWS_KEPT || p.num_splits == 1) {
          // the caller's rows hold d_io <= D columns (multiples of 8); only
          // the 128-wide kernel serves padded head dims
          const int d_io = (D == 64) ? D : p.d_io;
          if (32 * c >= d_io) continue;
          store_row32(p.o + row_off * d_io + 32 * c, v, min(4, (d_io - 32 * c) / 8), p.wide_out);
        } else {
          float4* dst = reinterpret_cast<float4*>(
              p.o_part + (static_cast<size_t>(split) * p.BH * p.rows_q + row_off) * D + 32 * c);
#pragma unroll
          for (int k = 0; k < 8; ++k) dst[k] = make_float4(v[4 * k], v[4 * k + 1], v[4 * k + 2], v[4 * k + 3]);
        }
      } else if (t < qt_n) {
        // (an empty tile's warps skip the O wait: they must not touch the
        // stages, which the other tile's MMAs may still be reading)
        // row row_local of box c: 16-byte piece k at piece k ^ (row mod 8)
        uint8_t* box_row = smem + L::OFF_K + (t * (D / 32) + c) * kBoxBytes + row_local * 128;
#pragma unroll
        for (int k = 0; k < 8; ++k)
          *reinterpret_cast<float4*>(box_row + ((k ^ (row_local & 7)) << 4)) =
              make_float4(v[4 * k], v[4 * k + 1], v[4 * k + 2], v[4 * k + 3]);
      }
    }
    if (SPLIT && t < qt_n) {  // a tile past the rows stores nothing
      fence_proxy_async_smem();  // the TMA unit reads the boxes next
      // this tile's four warps (barrier 1 or 2; 0 is __syncthreads)
      if (t == 0)
        named_barrier_sync<1, 4 * 32>();
      else
        named_barrier_sync<2, 4 * 32>();
      if (wq == 0 && lane == 0) {
        const uint8_t* stage = smem + L::OFF_K + t * (D / 32) * kBoxBytes;
#pragma unroll
        for (int c = 0; c < (DM + 31) / 32; ++c)
          tma_store_3d(&tm_op, stage + c * kBoxBytes, 32 * c, r0 + t * kTileRows, split * p.BH + bh);
        bulk_commit_group();
        bulk_wait_read<0>();  // the boxes are read before the CTA's shared memory goes
      }
    }
    if (row_valid) {
      if constexpr (!SPLIT) {
        if (p.lse) p.lse[row_off] = lse;
      } else {
        p.lse_part[static_cast<size_t>(split) * p.BH * p.rows_q + row_off] = lse;
      }
    }
  }

  __syncwarp();
  tc_fence_before();
  __syncthreads();
  if (warp == 9) {
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
}

// Merge of split-KV partials (per row): LSE = ln sum_s exp(LSE_s),
// O = sum_s exp(LSE_s - LSE) O_s.  D / 8 lanes per row, 8 columns each: the
// partials come from L2, so bytes in flight bound it, and a launch has few rows
// (more splits, fewer rows), so a lane takes one row and issues all its loads
// before it uses the first (S splits, 2 to 8; S = 0: any number, eight at a
// time).  A step (forward and combine), us, with two rows a lane and one split
// after another from five splits on -> this form: 8 heads of 64, 200 new rows,
// five splits against one chunk 11.1 -> 7.6, eleven against twelve chunks 15.6
// -> 9.8; 12 of 128, 440 rows, five splits 16.1 -> 13.2; 12 of 128, 880 rows,
// three splits 17.9 -> 17.7; 16 of 128, 880 rows, two splits 20.9 -> 20.5.  (A
// warp a row with one 16-byte load a split: 8.7, 11.6, 14.5, 19.4 and 20.7.)
// The blocks after those of the rows carry the ring commit cj (one thread per
// 16-byte piece of a committed row of one head), when there is one.
template <int D, int S>
__global__ void __launch_bounds__(256) combine_kernel(const float* __restrict__ o_part,
                                                      const float* __restrict__ lse_part,
                                                      __nv_bfloat16* __restrict__ o,
                                                      float* __restrict__ lse, int splits,
                                                      int n_rows, int d_io_arg,
                                                      const CommitJob cj) {
  pdl_wait();     // the forward's partials (and its reads of the ring) are complete
  pdl_trigger();  // the next step's forward may start its setup meanwhile
  constexpr int G = D / 8;  // lanes per row
  constexpr int kBlockRows = 256 / G;
  const int combine_blocks = (n_rows + kBlockRows - 1) / kBlockRows;
  if (static_cast<int>(blockIdx.x) >= combine_blocks) {
    const long long idx =
        static_cast<long long>(blockIdx.x - combine_blocks) * blockDim.x + threadIdx.x;
    const int per_head = cj.rows * (cj.d / 8);
    if (idx < static_cast<long long>(per_head) * cj.BH)
      commit_piece(cj, static_cast<int>(idx / per_head), static_cast<int>(idx % per_head));
    return;
  }
  const int d_io = (D == 64) ? D : d_io_arg;  // padded head dims use the 128-wide kernels
  const int sub = threadIdx.x % G;
  const int row = blockIdx.x * kBlockRows + threadIdx.x / G;
  // (the multiples of 8 columns past the caller's hold nothing)
  if (8 * sub >= d_io) return;
  constexpr int kAll = S > 0 ? S : kMaxSplits;
  constexpr int kChunk = S > 0 ? S : 8;  // splits whose columns are in registers at once
  const int n = S > 0 ? S : splits;
  const size_t split_stride = static_cast<size_t>(n_rows) * D;
  float ls[kAll], acc[8], m = -INFINITY, wsum = 0.f;
  float4 x[kChunk][2];
#pragma unroll
  for (int k = 0; k < 8; ++k) acc[k] = 0.f;
#pragma unroll
  for (int s = 0; s < kAll; ++s)
    if (s < n && row < n_rows) ls[s] = lse_part[static_cast<size_t>(s) * n_rows + row];
#pragma unroll
  for (int s0 = 0; s0 < kAll; s0 += kChunk) {
    if (s0 >= n) break;
#pragma unroll
    for (int k = 0; k < kChunk; ++k)
      if (s0 + k < n && row < n_rows) {
        const float4* src = reinterpret_cast<const float4*>(
            o_part + (s0 + k) * split_stride + static_cast<size_t>(row) * D + 8 * sub);
        x[k][0] = src[0];
        x[k][1] = src[1];
      }
    // (tested again here, and not left early above: with both parts in one
    // block the compiler moves each load next to its use)
    if (row >= n_rows) break;
    if (s0 == 0) {
#pragma unroll
      for (int s = 0; s < kAll; ++s)
        if (s < n) m = fmaxf(m, ls[s]);
    }
    // a split whose LSE is -inf saw no key of the row: its O part is skipped
    // (never multiplied: it may hold anything)
#pragma unroll
    for (int k = 0; k < kChunk; ++k) {
      if (s0 + k >= n) break;
      const float w = ls[s0 + k] == -INFINITY ? 0.f : __expf(ls[s0 + k] - m);
      wsum += w;
      if (w > 0.f) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          acc[4 * h] += w * x[k][h].x;
          acc[4 * h + 1] += w * x[k][h].y;
          acc[4 * h + 2] += w * x[k][h].z;
          acc[4 * h + 3] += w * x[k][h].w;
        }
      }
    }
  }
  if (row >= n_rows) return;
  const float inv = wsum > 0.f ? 1.f / wsum : 0.f;
  *reinterpret_cast<uint4*>(o + static_cast<size_t>(row) * d_io + 8 * sub) =
      make_uint4(pack_bf16x2(acc[0] * inv, acc[1] * inv), pack_bf16x2(acc[2] * inv, acc[3] * inv),
                 pack_bf16x2(acc[4] * inv, acc[5] * inv), pack_bf16x2(acc[6] * inv, acc[7] * inv));
  if (lse && sub == 0) lse[row] = wsum > 0.f ? m + __logf(wsum) : -INFINITY;
}

template <int D, int DM, bool ROPE, bool SPLIT>
cudaError_t launch_fwd_t(const CUtensorMap& tq, const CUtensorMap& tk, const CUtensorMap& tv,
                         const CUtensorMap& tkr, const CUtensorMap& tvr, const CUtensorMap& tks,
                         const CUtensorMap& tvs, const CUtensorMap& top, const FwdParams& p,
                         const RopeFreq& om, int dev, cudaStream_t s) {
  using L = FwdLayout<D, DM, ROPE, SPLIT>;
  static OncePerDevice prepared;
  const cudaError_t e = prepared(dev, [] {
    // The in-kernel register re-split assumes the launch register count; with
    // any other count its setmaxnreg.inc could never be satisfied, so refuse.
    cudaFuncAttributes fa;
    const cudaError_t e0 = cudaFuncGetAttributes(&fa, bca_fwd_kernel<D, DM, ROPE, SPLIT>);
    if (e0 != cudaSuccess) return e0;
    if (fa.numRegs != L::REGS_LAUNCH) return cudaErrorInvalidKernelImage;
    return cudaFuncSetAttribute(bca_fwd_kernel<D, DM, ROPE, SPLIT>,
                                cudaFuncAttributeMaxDynamicSharedMemorySize, L::BYTES);
  });
  if (e != cudaSuccess) return e;
  const unsigned grid = static_cast<unsigned>(p.BH) * p.n_qblocks * p.num_splits;
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr;
  pdl_config(cfg, attr, dim3(grid), dim3(L::THREADS), L::BYTES, s);
  return cudaLaunchKernelEx(&cfg, bca_fwd_kernel<D, DM, ROPE, SPLIT>, tq, tk, tv, tkr, tvr, tks, tvs, top, p,
                            om);
}

template <bool SPLIT>
cudaError_t launch_fwd_split(int d, int dm, const CUtensorMap& tq, const CUtensorMap& tk,
                             const CUtensorMap& tv, const CUtensorMap& tkr, const CUtensorMap& tvr,
                             const CUtensorMap& tks, const CUtensorMap& tvs, const CUtensorMap& top,
                             const FwdParams& p, const RopeFreq& om, int dev, cudaStream_t s) {
  if (p.rope_dims > 0) {
    if (d == 64) return launch_fwd_t<64, 64, true, SPLIT>(tq, tk, tv, tkr, tvr, tks, tvs, top, p, om, dev, s);
    if (dm == 80) return launch_fwd_t<128, 80, true, SPLIT>(tq, tk, tv, tkr, tvr, tks, tvs, top, p, om, dev, s);
    return launch_fwd_t<128, 128, true, SPLIT>(tq, tk, tv, tkr, tvr, tks, tvs, top, p, om, dev, s);
  }
  if (d == 64) return launch_fwd_t<64, 64, false, SPLIT>(tq, tk, tv, tkr, tvr, tks, tvs, top, p, om, dev, s);
  if (dm == 80) return launch_fwd_t<128, 80, false, SPLIT>(tq, tk, tv, tkr, tvr, tks, tvs, top, p, om, dev, s);
  return launch_fwd_t<128, 128, false, SPLIT>(tq, tk, tv, tkr, tvr, tks, tvs, top, p, om, dev, s);
}

}  // namespace

cudaError_t launch_fwd(int d, int dm, const CUtensorMap& tq, const CUtensorMap& tk, const CUtensorMap& tv,
                       const CUtensorMap& tkr, const CUtensorMap& tvr, const CUtensorMap& tks,
                       const CUtensorMap& tvs, const CUtensorMap& top, const FwdParams& p,
                       const RopeFreq& om, int dev, cudaStream_t s) {
  return p.num_splits > 1 ? launch_fwd_split<true>(d, dm, tq, tk, tv, tkr, tvr, tks, tvs, top, p, om, dev, s)
                          : launch_fwd_split<false>(d, dm, tq, tk, tv, tkr, tvr, tks, tvs, top, p, om, dev, s);
}

cudaError_t launch_combine(int d, int d_io, const float* o_part, const float* lse_part,
                           __nv_bfloat16* o, float* lse, int splits, int BH, int rows,
                           const CommitJob& cj, cudaStream_t s) {
  const int n_rows = BH * rows;
  const long long commit_pieces = static_cast<long long>(cj.rows) * (cj.d / 8) * cj.BH;
  const int block_rows = 256 / (d / 8);
  const long long blocks = (n_rows + block_rows - 1) / block_rows + (commit_pieces + 255) / 256;
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr;
  pdl_config(cfg, attr, dim3(static_cast<unsigned>(blocks)), dim3(256), 0, s);
  auto launch = [&](auto kernel) {
    return cudaLaunchKernelEx(&cfg, kernel, o_part, lse_part, o, lse, splits, n_rows, d_io, cj);
  };
  auto by_splits = [&](auto width) {
    constexpr int D = decltype(width)::value;
    switch (splits) {
      case 2: return launch(combine_kernel<D, 2>);
      case 3: return launch(combine_kernel<D, 3>);
      case 4: return launch(combine_kernel<D, 4>);
      case 5: return launch(combine_kernel<D, 5>);
      case 6: return launch(combine_kernel<D, 6>);
      case 7: return launch(combine_kernel<D, 7>);
      case 8: return launch(combine_kernel<D, 8>);
      default: return launch(combine_kernel<D, 0>);
    }
  };
  return d == 64 ? by_splits(std::integral_constant<int, 64>{}) : by_splits(std::integral_constant<int, 128>{});
}

}  // namespace mw
