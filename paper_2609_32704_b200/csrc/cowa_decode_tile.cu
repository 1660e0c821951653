// Decode of several tokens per sequence and / or over a paged cache (the forward with N_q = Nq and N_k = lens[b]).
//
// All Nq tokens x G heads that share a KV head are the rows of one 128-row tile, so that every visible cache row is
// read once: S = Q K^T and O += P V run on tcgen05 with 64-key steps, K and V arrive by TMA (whole 64-row tiles of a
// contiguous cache, 16- to 64-row boxes of its pages).  The 64-key tiles of all units -- a unit is (sequence, KV head,
// row tile) -- form one list that is cut into equal shares, one per resident block (two per SM), so that sequences of
// very different lengths still end together.  A block's share is a run of pieces of consecutive units; a piece leaves its
// row states (reference max, sum, un-normalised O, fp32) in the workspace and a second kernel merges a unit's pieces.
// Bound by HBM: 32 KB per step; two blocks per SM take a step in about 1600 clocks each, twice the rate at which HBM
// feeds them.
// Warps 0-3: softmax, one row per thread (only as many warps as there are rows); warp 4: TMA; warp 5: MMA issue.  V rows
// that no token sees are cleared by the warps without rows beside the softmax, by all four when each of them has rows
// (a warp of its own would leave the threads 128 registers, and they spill).
#include <cuda_bf16.h>
#include <string.h>

#include <algorithm>

#include "cowa_common.h"
#include "cowa_ptx.cuh"
#include "cowa_tma.h"

using namespace cowa_ptx;

namespace {

constexpr int BQ = 128, BK = 64;
constexpr int kThreads = 192;

struct TileArgs {
  const int32_t* lens;
  const int32_t* block_table;  // [B, max_pages], or nullptr: contiguous cache
  float* ws_o;                 // [slots, rows, D]
  float2* ws_ml;               // [slots, rows]
  int2* ws_unit;               // [units] first block of the unit's pieces, number of pieces
  unsigned int* status;
  int B, Nq, Hq, Hkv, G;
  int tpt, ntiles, rows;       // tokens per row tile, row tiles per (sequence, KV head), rows of a full tile
  int units;
  int page_size, max_pages, box;  // box: cache rows per TMA load of a page
  int sink, local, hkv_global, hkv_offset, full_attn;
  float scale_log2;
};

// A unit's geometry.
struct Unit {
  int b, hk, tok0, tok1, Nk, off;  // tokens [tok0, tok1), token t at key position off + t
  CowaWin w;
  CowaRange rg[3];
  int nt;  // visited 64-key tiles
};

__device__ __forceinline__ int length_of(const TileArgs& a, int u) { return a.lens[u / (a.ntiles * a.Hkv)]; }
__device__ __forceinline__ void unit_of(const TileArgs& a, int u, int Nk, Unit& x) {  // Nk: length_of(a, u)
  const int tile = u % a.ntiles;
  const int bh = u / a.ntiles;
  x.hk = bh % a.Hkv; x.b = bh / a.Hkv;
  x.Nk = Nk;
  x.off = x.Nk - a.Nq;
  x.tok0 = tile * a.tpt; x.tok1 = min(x.tok0 + a.tpt, a.Nq);
  if (a.full_attn) { x.w.s = 0; x.w.n = x.Nk; x.w.g = 0; x.w.l = 0; }
  else x.w = cowa_default_window(x.Nk, a.hkv_global, a.hkv_offset + x.hk, a.sink, a.local);
  cowa_fwd_ranges(x.w, x.tok0, x.tok1 - 1, x.off, x.Nk, BK, x.rg);
  x.nt = cowa_range_len(x.rg[0]) + cowa_range_len(x.rg[1]) + cowa_range_len(x.rg[2]);
}

// A piece of a unit as the TMA warp publishes it.
struct Piece {
  Unit u;
  int f_lo[3], f_hi[3];  // tiles that need no mask, one interval per range
  int t0, n;             // steps t0 .. t0 + n - 1 of the unit; n = 0: no more pieces
  int slot;
};
static_assert(sizeof(Piece) <= 128, "slot of a published piece");

// Key tile of step t of a piece, and whether every token sees all of it.
__device__ __forceinline__ int tile_of(const Piece& pc, int t, bool* full) {
  const int i = pc.t0 + t, n0 = cowa_range_len(pc.u.rg[0]), n1 = n0 + cowa_range_len(pc.u.rg[1]);
  const int j = i < n0 ? pc.u.rg[0].hi - i : i < n1 ? pc.u.rg[1].hi + n0 - i : pc.u.rg[2].hi + n1 - i;
  const int lo = i < n0 ? pc.f_lo[0] : i < n1 ? pc.f_lo[1] : pc.f_lo[2];
  const int hi = i < n0 ? pc.f_hi[0] : i < n1 ? pc.f_hi[1] : pc.f_hi[2];
  *full = j >= lo && j <= hi;
  return j;
}

// The keys that tokens at key positions p0 .. p1 (p0 >= 0) see, some of them (first = p0, last = p1) or each of them by
// the same window (first = p1, last = p0), in the 64 keys from `row0` on: one bit per key.
__device__ __forceinline__ unsigned long long seen_bits(const CowaWin& w, int first, int last, int row0) {
  uint32_t m[2];
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const int base = row0 + q * 32;
    m[q] = interval_bits(max(first - w.n + 1, 0), last, base) | interval_bits(0, min(w.s - 1, last), base);
    if (w.l > 0) m[q] |= interval_bits(first - (w.n + w.g + w.l) + 1, last - (w.n + w.g), base);
  }
  return (unsigned long long)m[1] << 32 | m[0];
}
// Keys of a unit that some token sees.  Other rows of the cache are nobody's: they may be stale, non-finite, or lie in pages
// that were handed to somebody else.
__device__ __forceinline__ unsigned long long seen_by_some(const Unit& u, int row0) {
  return seen_bits(u.w, max(u.off + u.tok0, 0), u.off + u.tok1 - 1, row0);
}
__device__ __forceinline__ unsigned long long seen_by_all(const Unit& u, int row0) {
  return seen_bits(u.w, u.off + u.tok1 - 1, max(u.off + u.tok0, 0), row0);
}

// QR rows of Q and NS slots each for K and V: 128 and 2, or, when a tile has at most 32 rows (S and O of the other rows
// of the MMA are then computed from whatever lies behind Q and never read), 32 and 3.
template <int D, int QR, int NS>
struct TileSmem {
  static constexpr int kQ = QR * D * 2, kKV = BK * D * 2;
  static constexpr int oQ = 0, oK = kQ, oV = oK + NS * kKV, oBar = oV + NS * kKV, oPiece = oBar + 256, oScan = oPiece + 256;
  static constexpr int kBytes = oScan + 64 + 1024;  // + alignment slack
};

// a pair of bf16 holds an Inf or a NaN
__device__ __forceinline__ bool nonfinite(uint32_t x) { return (x & 0x7F80u) == 0x7F80u || (x & 0x7F800000u) == 0x7F800000u; }

// O += P V of one step on the FMA pipe, each row over the keys it sees (mk): for tiles whose V holds an Inf or a NaN.
template <int D>
__device__ __forceinline__ void add_seen(const uint8_t* vt, uint32_t t_P, uint32_t t_O, unsigned long long mk) {
#pragma unroll 1
  for (int q = 0; q < D / 16; ++q) {
    uint32_t ov[16], pw;
    tmem_ld16(t_O + q * 16, ov);
#pragma unroll 1
    for (int r = 0; r < BK; ++r) {
      tmem_ld1(t_P + (r >> 1), pw);
      tmem_wait_ld();
      const float p = __uint_as_float(r & 1 ? pw & 0xFFFF0000u : pw << 16);
      const uint8_t* row = vt + (q >> 2) * (BK * 128) + r * 128;
      const bool sees = (mk >> r) & 1ull;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const uint4 x = *reinterpret_cast<const uint4*>(row + ((((q & 3) * 2 + h) ^ (r & 7)) << 4));
        const uint32_t xs[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          const float y = __uint_as_float(e & 1 ? xs[e >> 1] & 0xFFFF0000u : xs[e >> 1] << 16);
          const float o = __uint_as_float(ov[h * 8 + e]);
          ov[h * 8 + e] = __float_as_uint(sees ? fmaf(p, y, o) : o);
        }
      }
    }
    tmem_st16(t_O + q * 16, ov);
  }
  tmem_wait_st();
}

template <int D, int QR, int NS>
__global__ void __launch_bounds__(kThreads, 2)
cowa_decode_tile_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                        const __grid_constant__ CUtensorMap tmV, const __grid_constant__ TileArgs a) {
  using SM = TileSmem<D, QR, NS>;
  constexpr int NSLAB = D / 64;
  constexpr int SLAB_Q = QR * 128, SLAB_K = BK * 128;
  constexpr uint32_t TMEM_COLS = 256, cO = 128;  // S/P buffers: [0,64), [64,128); O: [128, 128 + D)
  constexpr uint32_t IDESC_S = idesc_bf16(128, BK, 0, 0), IDESC_O = idesc_bf16(128, D, 0, 1);

  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* sQ = smem + SM::oQ;
  uint8_t* sK = smem + SM::oK;  // [NS][kKV]
  uint8_t* sV = smem + SM::oV;  // [NS][kKV]
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + SM::oBar);
  uint64_t* bar_q_full = bars + 0;    //     Q of a piece has landed
  uint64_t* bar_q_empty = bars + 1;   //     every S of the piece has been computed
  uint64_t* bar_pv = bars + 2;        //     O += P V of a step has completed
  uint64_t* bar_s = bars + 3;         // [2] S of a step is in TMEM buffer b
  uint64_t* bar_i_full = bars + 5;    // [2] a piece has been published
  uint64_t* bar_i_empty = bars + 7;   // [2] count 5 (warps 0-3, MMA): it has been read
  uint64_t* bar_p = bars + 9;         // [2] count nw: P written over S
  uint64_t* bar_v_read = bars + 11;   //     count nw: add_seen has read a V tile
  uint64_t* bar_k_full = bars + 12;             // [NS]
  uint64_t* bar_k_empty = bar_k_full + NS;      // [NS]
  uint64_t* bar_v_full = bar_k_full + 2 * NS;   // [NS]
  uint64_t* bar_v_empty = bar_k_full + 3 * NS;  // [NS]
  uint64_t* bar_v_seen = bar_k_full + 4 * NS;   // [NS] count 4 - nw, or 4: V rows that no token sees are cleared
  uint64_t* bar_v_go = bar_k_full + 5 * NS;     // [NS] V of a boundary tile is on its way (the clearing warps pass other steps by)
  uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(bar_k_full + 6 * NS);
  int* scan = reinterpret_cast<int*>(smem + SM::oScan);  // 6 warp totals; [8], [9] first unit and its list position; [10 ..] per slot: step whose V is not finite

  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);  // warp-uniform by construction
  const int nw = (a.rows + 31) >> 5;                       // softmax warps with rows

  if (tid == 128) { prefetch_tmap(&tmQ); prefetch_tmap(&tmK); prefetch_tmap(&tmV); }
  if (tid == 0) {
    for (int s = 0; s < 12 + 6 * NS; ++s) {
      const bool v_seen = bars + s >= bar_v_seen && bars + s < bar_v_go;
      mbar_init(bars + s, s == 7 || s == 8 ? 5 : s >= 9 && s < 12 ? nw : !v_seen ? 1 : nw < 4 ? 4 - nw : 4);
    }
    for (int s = 0; s < NS; ++s) scan[10 + s] = 0;
    fence_mbar_init();
  }
  grid_enter();  // the merge kernel's blocks may be scheduled beside this one's; they wait for its results
  if (warp == 5) {
    __syncwarp();
    tmem_alloc(tmem_holder, TMEM_COLS);
    tmem_relinquish();
  }

  // ---- this block's share of the list of all units' steps ----
  // Every instruction here delays the first load of K.  A thread works out two units at a time, side by side (their divisions are long
  // chains), keeps the step counts of the first two, and the block's first unit is handed on as it was worked out.  (One unit
  // after the other, found and handed on by its number, with 64-bit divisions: 2.9 us for 256 units, so 1.6.)
  const int per = (a.units + kThreads - 1) / kThreads;
  const int u_lo = min(tid * per, a.units), u_hi = min(u_lo + per, a.units);
  Unit first[2];  // of this thread
  int sum = 0;
  for (int u0 = u_lo; u0 < u_hi; u0 += 2) {
    Unit x[2];
    const int len0 = length_of(a, u0), len1 = length_of(a, min(u0 + 1, a.units - 1));
    unit_of(a, u0, len0, x[0]);
    unit_of(a, min(u0 + 1, a.units - 1), len1, x[1]);
    sum += x[0].nt + (u0 + 1 < u_hi ? x[1].nt : 0);
    if (u0 == u_lo) { first[0] = x[0]; first[1] = x[1]; }
  }
  int incl = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
    if (lane >= o) incl += y;
  }
  if (lane == 31) scan[warp] = incl;
  __syncthreads();
  int base = 0, total = 0;
#pragma unroll
  for (int i = 0; i < kThreads / 32; ++i) {
    if (i < warp) base += scan[i];
    total += scan[i];
  }
  const int nb = min((int)gridDim.x, total);  // no share is empty: the merge expects a piece from every block of a run
  const bool mine = (int)blockIdx.x < nb;
  const int lo = mine ? (int)((long long)blockIdx.x * total / nb) : 0;
  const int hi = mine ? (int)((long long)(blockIdx.x + 1) * total / nb) : 0;
  const int excl = base + incl - sum;
  if (lo < hi && excl <= lo && lo < excl + sum) {
    int f = excl, u = u_lo;
    Unit x = first[0];
    if (lo >= f + x.nt) {
      f += x.nt; ++u;
      x = first[1];
      while (lo >= f + x.nt) {  // (more than two units a thread)
        f += x.nt; ++u;
        unit_of(a, u, length_of(a, u), x);
      }
    }
    *reinterpret_cast<Unit*>(smem + SM::oPiece + 128) = x;  // (the slot of the second piece)
    scan[8] = u; scan[9] = f;
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tb = *tmem_holder;

  bool ok = true;  // false once a bounded wait ran out; every role then falls through to the teardown
  auto warp_arrive = [&](uint64_t* bar) {
    __syncwarp();
    if (lane == 0) mbar_arrive(bar);
  };
  // Piece number ni of this block (its words go through a shuffle: uniform for the compiler); false: none left.
  auto next_piece = [&](uint32_t ni, Piece& pc) -> bool {
    ok = mbar_wait(bar_i_full + (ni & 1), (ni >> 1) & 1, a.status);
    if (!ok) return false;
    const int* src = reinterpret_cast<const int*>(smem + SM::oPiece + (ni & 1) * 128);
    int words[sizeof(Piece) / 4];
#pragma unroll
    for (int i = 0; i < (int)(sizeof(Piece) / 4); ++i) words[i] = __shfl_sync(0xFFFFFFFFu, src[i], 0);
    warp_arrive(bar_i_empty + (ni & 1));
    memcpy(&pc, words, sizeof(Piece));
    return pc.n > 0;
  };

  // Boundary tiles, once V is in `slot`: clears the rows that no token sees and looks through those that not every token
  // sees; scan[10 + slot] becomes c + 1 (of step c) when one of these holds an Inf or a NaN.  Warp wi of n.
  auto clear_unseen = [&](const Unit& u, int j, int slot, int c, int wi, int n) {
    constexpr int CPR = D / 8, RPI = 32 / CPR;  // 16-byte chunks per row, rows per pass of a warp
    const int ch = lane % CPR;
    const unsigned long long some = seen_by_some(u, j * BK), all = seen_by_all(u, j * BK);
    uint8_t* vt = sV + slot * SM::kKV + (ch >> 3) * SLAB_K;
    bool bad = false;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const uint32_t look = ~(uint32_t)(all >> (32 * h)), keep = (uint32_t)(some >> (32 * h));
      if (look == 0u) continue;
#pragma unroll 4
      for (int r = wi * RPI + lane / CPR; r < 32; r += n * RPI) {
        if (!((look >> r) & 1u)) continue;
        uint4* x = reinterpret_cast<uint4*>(vt + (h * 32 + r) * 128 + (((ch & 7) ^ (r & 7)) << 4));
        if (!((keep >> r) & 1u)) {
          *x = make_uint4(0u, 0u, 0u, 0u);
        } else {
          const uint4 y = *x;
          bad = bad || nonfinite(y.x) || nonfinite(y.y) || nonfinite(y.z) || nonfinite(y.w);
        }
      }
    }
    fence_proxy_async_smem();
    if (__any_sync(0xFFFFFFFFu, bad) && lane == 0) *(volatile int*)(scan + 10 + slot) = c + 1;
    warp_arrive(bar_v_seen + slot);
  };

  if (warp == 4) {
    // ======================= TMA producer =======================
    const bool lead = elect_one();
    int sl = 0;         // slot of the next step's K and V
    uint32_t rnd = 0;   // times the slots have been gone through
    uint32_t ni = 0;    // pieces so far
    int pos = lo, u = lo < hi ? scan[8] : 0, f = lo < hi ? scan[9] : 0;
    Unit unit;  // u
    if (lo < hi) unit = *reinterpret_cast<const Unit*>(smem + SM::oPiece + 128);
    __syncwarp();
    int Nk = 0;  // length of unit u, where `unit` has not been worked out
    bool have = true;
    while (ok) {
      Piece pc;
      pc.n = 0;
      if (pos < hi) {
        if (have) pc.u = unit;
        else unit_of(a, u, Nk, pc.u);
        have = false;
        Nk = length_of(a, min(u + 1, a.units - 1));  // of the next one, before it is needed
        if (pc.u.nt == 0) { ++u; continue; }
        pc.t0 = pos - f;
        pc.n = min(pc.u.nt, hi - f) - pc.t0;
        pc.slot = blockIdx.x + u;
        const CowaWin w = pc.u.w;
        auto fdiv = [](long long v) -> int { return (int)(v >> 6); };  // floor of v / BK
        const long long p0 = (long long)pc.u.off + pc.u.tok0, p1 = (long long)pc.u.off + pc.u.tok1 - 1;
        const int causal_hi = fdiv(p0 - (BK - 1));
        pc.f_lo[0] = fdiv(p1 - w.n) + 1; pc.f_hi[0] = causal_hi;
        pc.f_lo[1] = 1; pc.f_hi[1] = 0;
        if (w.l > 0) {
          pc.f_lo[1] = fdiv(p1 - ((long long)w.n + w.g + w.l)) + 1;
          pc.f_hi[1] = min(causal_hi, fdiv(p0 - ((long long)w.n + w.g) - (BK - 1)));
        }
        pc.f_lo[2] = 0; pc.f_hi[2] = min(causal_hi, w.s >= BK ? (w.s - BK) / BK : -1);
        if (pc.t0 == 0 && lead) {  // the unit begins here: its pieces lie in this block and the following ones
          const long long last = f + pc.u.nt - 1;
          a.ws_unit[u] = make_int2(blockIdx.x, (int)(((last + 1) * nb - 1) / total) - (int)blockIdx.x + 1);
        }
      }
      if (ni >= 2) ok = mbar_wait(bar_i_empty + (ni & 1), ((ni >> 1) & 1) ^ 1, a.status);
      if (!ok) break;
      if (lead) {
        *reinterpret_cast<Piece*>(smem + SM::oPiece + (ni & 1) * 128) = pc;
        mbar_arrive(bar_i_full + (ni & 1));
      }
      __syncwarp();
      if (pc.n == 0) break;

      // One 64-row tile.  Paged cache: every lane looks up the page of its box (box rows of one page) and loads it; boxes
      // without a key that a token sees are left out (their table entries may be anything): page -1.
      const int boxes = a.block_table ? BK / a.box : 1;
      auto page_of = [&](int t) -> int {
        const int row0 = cowa_fwd_tile_at(pc.u.rg, pc.t0 + t) * BK, row = row0 + lane * a.box;
        const unsigned long long box_mask = (a.box == 64 ? ~0ull : (1ull << a.box) - 1) << (lane * a.box & 63);
        if (lane >= boxes || !(seen_by_some(pc.u, row0) & box_mask)) return -1;
        return max(a.block_table[(size_t)pc.u.b * a.max_pages + row / a.page_size], 0);
      };
      auto load = [&](uint8_t* dst, const CUtensorMap* tm, uint64_t* bar, int t, int page) {
        const int row0 = cowa_fwd_tile_at(pc.u.rg, pc.t0 + t) * BK;
        if (!a.block_table) {
          if (lead) {
            mbar_expect_tx(bar, SM::kKV);
            for (int s = 0; s < NSLAB; ++s) tma_load_4d(dst + s * SLAB_K, tm, bar, s * 64, row0, pc.u.hk, pc.u.b);
          }
        } else {
          const unsigned live = __ballot_sync(0xFFFFFFFFu, page >= 0);
          if (lead) mbar_expect_tx(bar, __popc(live) * a.box * D * 2);
          __syncwarp();
          if (page >= 0)
            for (int s = 0; s < NSLAB; ++s)
              tma_load_4d(dst + s * SLAB_K + lane * a.box * 128, tm, bar, s * 64, (row0 + lane * a.box) % a.page_size, pc.u.hk,
                          page);
        }
      };
      int page = a.block_table ? page_of(0) : 0;  // this lane's page of the next tile
      for (int t = 0; t < pc.n; ++t) {
        if (rnd > 0) ok = mbar_wait(bar_k_empty + sl, (rnd - 1) & 1, a.status);
        if (!ok) break;
        load(sK + sl * SM::kKV, &tmK, bar_k_full + sl, t, page);
        if (t == 0) {
          if (ni > 0) ok = mbar_wait(bar_q_empty, (ni - 1) & 1, a.status);
          if (!ok) break;
          if (lead) {
            const int qrows = a.rows;  // G heads x tokens of a full tile: the box of the map
            mbar_expect_tx(bar_q_full, qrows * D * 2);
            for (int s = 0; s < NSLAB; ++s)
              tma_load_4d(sQ + s * SLAB_Q, &tmQ, bar_q_full, s * 64, pc.u.hk * a.G, pc.u.tok0, pc.u.b);
          }
        }
        const int next = a.block_table && t + 1 < pc.n ? page_of(t + 1) : 0;
        if (rnd > 0) ok = mbar_wait(bar_v_empty + sl, (rnd - 1) & 1, a.status);
        if (!ok) break;
        load(sV + sl * SM::kKV, &tmV, bar_v_full + sl, t, page);
        bool full;
        tile_of(pc, t, &full);
        if (lead && !full) mbar_arrive(bar_v_go + sl);
        page = next;
        if (++sl == NS) { sl = 0; ++rnd; }
      }
      pos = f + pc.t0 + pc.n;
      f += pc.u.nt;
      ++u;
      ++ni;
    }
  } else if (warp == 5) {
    // ======================= MMA issuer (warp-uniform control flow, one elected lane issues) =======================
    const bool lead = elect_one();
    const uint64_t dQ = smem_desc_sw128(smem_u32(sQ), 16, 1024);       // Q, K-major (A of S)
    const uint64_t dK0 = smem_desc_sw128(smem_u32(sK), 16, 1024);      // K, K-major (B of S)
    const uint64_t dV0 = smem_desc_sw128(smem_u32(sV), SLAB_K, 1024);  // V, MN-major (B of O)
    constexpr uint32_t kKV16 = SM::kKV >> 4;
    int c = 0;                  // steps so far: S buffer c & 1
    int ks = 0, vs = 0;         // slots of the next S and the next O += P V
    uint32_t kr = 0, vr = 0;    // parities of those slots' loads
    uint32_t ni = 0;
    Piece pc;
    for (; ok && next_piece(ni, pc); ++ni) {
      const int n = pc.n;
      auto issue_s = [&](int buf, bool last) {  // S of the next step into buffer `buf`, once its K has landed
        ok = mbar_wait(bar_k_full + ks, kr, a.status);
        if (!ok) return;
        tc_fence_after();
        if (lead) {
          const uint64_t dB = dK0 + ks * kKV16;
#pragma unroll
          for (int kk = 0; kk < D / 16; ++kk)
            mma_ss(tb + buf * 64, dQ + (((kk / 4) * SLAB_Q + (kk % 4) * 32) >> 4), dB + (((kk / 4) * SLAB_K + (kk % 4) * 32) >> 4),
                   IDESC_S, kk > 0);
          mma_commit(bar_s + buf);
          mma_commit(bar_k_empty + ks);
          if (last) mma_commit(bar_q_empty);
        }
        if (++ks == NS) { ks = 0; kr ^= 1; }
      };
      ok = mbar_wait(bar_q_full, ni & 1, a.status);
      if (!ok) break;
      issue_s(c & 1, n == 1);
      for (int t = 0; t < n && ok; ++t, ++c) {
        const int b_ = c & 1;
        if (t + 1 < n) issue_s(b_ ^ 1, t + 2 == n);  // its buffer last held P(c - 1), whose product was issued before
        ok = ok && mbar_wait(bar_v_full + vs, vr, a.status) && mbar_wait(bar_p + b_, (c >> 1) & 1, a.status);
        if (!ok) break;
        tc_fence_after();
        if (lead) {
          const uint64_t dB = dV0 + vs * kKV16;
#pragma unroll
          for (int kk = 0; kk < BK / 16; ++kk)
            mma_ts(tb + cO, tb + b_ * 64 + kk * 8, dB + ((kk * 2048) >> 4), IDESC_O, 1u);
          mma_commit(bar_pv);
          mma_commit(bar_v_empty + vs);
        }
        if (++vs == NS) { vs = 0; vr ^= 1; }
      }
    }
  } else if (warp < nw) {
    // ======================= softmax: one (token, head) row per thread =======================
    const uint32_t t_lane = tb + ((uint32_t)(warp * 32) << 16);
    const uint32_t t_O = t_lane + cO;
    const float2 sc2 = make_float2(a.scale_log2, a.scale_log2);
    int c = 0, vs = 0;    // steps so far; slot of this step's V
    uint32_t vr = 0;      // parity of its load
    uint32_t zr = 0;      // parities of bar_v_seen (bit per slot) and bar_v_read (bit 31)
    uint32_t ni = 0;
    Piece pc;
    for (; ok && next_piece(ni, pc); ++ni) {
      const int n = pc.n, Nk = pc.u.Nk;
      const int tok = pc.u.tok0 + tid / a.G;
      const bool row_valid = tid < a.rows && tok < pc.u.tok1;
      const int rowpos = pc.u.off + tok;  // position of this query on the key axis
      const CowaWin w = pc.u.w;
      float m_ref = -INFINITY, top = -INFINITY, l_sum = 0.f;
      {  // every product of the piece adds to O (the first one waits for this warp's P)
        uint32_t zero[16];
#pragma unroll
        for (int e = 0; e < 16; ++e) zero[e] = 0u;
#pragma unroll
        for (int q = 0; q < D / 16; ++q) tmem_st16(t_O + q * 16, zero);
      }

      for (int t = 0; t < n && ok; ++t, ++c) {
        const int b_ = c & 1;
        bool full;
        const int j = tile_of(pc, t, &full);
        const uint32_t t_S = t_lane + b_ * 64;

        ok = mbar_wait(bar_s + b_, (c >> 1) & 1, a.status);
        if (!ok) break;
        tc_fence_after();
        uint32_t sr[2][32];
        tmem_ld32(t_S, sr[0]);
        tmem_ld32(t_S + 32, sr[1]);
        tmem_wait_ld();
        uint32_t mk[2] = {0xFFFFFFFFu, 0xFFFFFFFFu};  // keys this row sees
        if (__builtin_expect(!full, 0)) {
          const int kend = row_valid ? min(rowpos, Nk - 1) : -1;  // last causal key of this row
          const int near_lo = rowpos - w.n + 1, sink_hi = min(w.s - 1, kend);
          const int long_hi = w.l > 0 ? min(rowpos - (w.n + w.g), kend) : -1, long_lo = rowpos - (w.n + w.g + w.l) + 1;
#pragma unroll
          for (int q = 0; q < 2; ++q) {
            const int base_ = j * BK + q * 32;
            mk[q] =
                interval_bits(near_lo, kend, base_) | interval_bits(0, sink_hi, base_) | interval_bits(long_lo, long_hi, base_);
#pragma unroll
            for (int e = 0; e < 32; ++e)
              if (!((mk[q] >> e) & 1u)) sr[q][e] = 0xFF800000u;  // -inf
          }
        }
        float mxa[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
        for (int q = 0; q < 2; ++q)
#pragma unroll
          for (int e = 0; e < 32; e += 2)
            mxa[(e >> 1) & 3] = max3(mxa[(e >> 1) & 3], __uint_as_float(sr[q][e]), __uint_as_float(sr[q][e + 1]));
        const float mx = fmaxf(fmaxf(mxa[0], mxa[1]), fmaxf(mxa[2], mxa[3])) * a.scale_log2;
        // The reference is every step's own maximum: the step's largest weight is then exactly 1 in bf16.  One that may lag by
        // 2^8 costs a tenth of the precision (o against 64 bits 0.0023 instead of 0.0021) for 1 us in 54.  A step far
        // below the largest so far keeps the reference: its weights do not count, and O stays in range.
        top = fmaxf(top, mx);
        const bool moved = row_valid && mx != m_ref && mx >= top - 16.f;
        const float alpha = moved ? ex2(m_ref - mx) : 1.f;
        if (moved) m_ref = mx;
        const float sub = (m_ref == -INFINITY) ? 0.f : m_ref;
        const float2 nsub2 = make_float2(-sub, -sub);
        float2 rsa[4] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
        uint32_t pk[32];
#pragma unroll
        for (int q = 0; q < 2; ++q)
#pragma unroll
          for (int e = 0; e < 32; e += 2) {
            const float2 y = fma2(make_float2(__uint_as_float(sr[q][e]), __uint_as_float(sr[q][e + 1])), sc2, nsub2);
            const float2 pp = make_float2(ex2(y.x), ex2(y.y));
            rsa[(e >> 1) & 3] = add2(rsa[(e >> 1) & 3], pp);
            pk[q * 16 + e / 2] = pack_bf16(pp.x, pp.y);
          }
        const float2 rs2 = add2(add2(rsa[0], rsa[1]), add2(rsa[2], rsa[3]));
        l_sum = l_sum * alpha + (rs2.x + rs2.y);
        // every step waits for the product of the step before: the accumulator may then be rescaled, and no thread
        // falls two phases behind on this barrier
        if (t > 0) {
          ok = mbar_wait(bar_pv, (c - 1) & 1, a.status);
          if (!ok) break;
          tc_fence_after();
          if (__any_sync(0xFFFFFFFFu, moved)) {
            const float2 al2 = make_float2(alpha, alpha);
#pragma unroll 1
            for (int q = 0; q < D / 16; ++q) {
              uint32_t ov[16];
              tmem_ld16(t_O + q * 16, ov);
              tmem_wait_ld();
#pragma unroll
              for (int e = 0; e < 16; e += 2) {
                const float2 y = mul2(make_float2(__uint_as_float(ov[e]), __uint_as_float(ov[e + 1])), al2);
                ov[e] = __float_as_uint(y.x); ov[e + 1] = __float_as_uint(y.y);
              }
              tmem_st16(t_O + q * 16, ov);
            }
          }
        }
        tmem_st32(t_S, pk);  // P over the first 32 columns of this S buffer
        tmem_wait_st();
        // P is exactly zero where a row does not see a key, but 0 x (Inf or NaN) in the product would not be: V rows that
        // no token sees have been cleared; where a row that some see holds such a value, every row takes the
        // keys it sees in add_seen, and the product gets zeros.
        if (__builtin_expect(!full, 0)) {
          if (nw == 4) {
            ok = mbar_wait(bar_v_full + vs, vr, a.status);
            if (!ok) break;
            clear_unseen(pc.u, j, vs, c, warp, 4);
          }
          ok = mbar_wait(bar_v_seen + vs, (zr >> vs) & 1, a.status);
          if (!ok) break;
          zr ^= 1u << vs;
          if (__builtin_expect(*(volatile int*)(scan + 10 + vs) == c + 1, 0)) {
            uint8_t* vt = sV + vs * SM::kKV;
            __syncwarp();
            add_seen<D>(vt, t_S, t_O, (unsigned long long)mk[1] << 32 | mk[0]);
            warp_arrive(bar_v_read);
            ok = mbar_wait(bar_v_read, zr >> 31, a.status);
            if (!ok) break;
            zr ^= 1u << 31;
            for (int c_ = tid; c_ < SM::kKV / 16; c_ += nw * 32)
              *reinterpret_cast<uint4*>(vt + c_ * 16) = make_uint4(0u, 0u, 0u, 0u);
            fence_proxy_async_smem();
          }
        }
        tc_fence_before();
        warp_arrive(bar_p + b_);
        if (++vs == NS) { vs = 0; vr ^= 1; }
      }
      if (!ok) break;

      // ---- the piece's row states ----
      ok = mbar_wait(bar_pv, (c - 1) & 1, a.status);
      if (!ok) break;
      tc_fence_after();
      const size_t srow = (size_t)pc.slot * a.rows + tid;
#pragma unroll 2
      for (int q = 0; q < D / 16; ++q) {
        uint32_t ov[16];
        tmem_ld16(t_O + q * 16, ov);
        tmem_wait_ld();
        if (row_valid) {
          uint4* dst = reinterpret_cast<uint4*>(a.ws_o + srow * D + q * 16);
#pragma unroll
          for (int e = 0; e < 4; ++e) dst[e] = make_uint4(ov[e * 4], ov[e * 4 + 1], ov[e * 4 + 2], ov[e * 4 + 3]);
        }
      }
      if (row_valid) a.ws_ml[srow] = make_float2(m_ref, l_sum);
    }
  } else if (warp < 4) {
    // ======================= boundary tiles, beside fewer than four softmax warps =======================
    // The TMA warp says when a tile of its kind is on its way: these warps pass the other steps by, and a wait for V alone
    // could meet the slot's load of two rounds before, which has the same parity.
    int c = 0, vs = 0;
    uint32_t vr = 0, gr = 0;  // parity of the slot's load; parities of bar_v_go, a bit per slot
    Piece pc;
    for (uint32_t ni = 0; ok && next_piece(ni, pc); ++ni) {
      for (int t = 0; t < pc.n; ++t, ++c) {
        bool full;
        const int j = tile_of(pc, t, &full);
        if (!full) {
          ok = mbar_wait(bar_v_go + vs, (gr >> vs) & 1, a.status) && mbar_wait(bar_v_full + vs, vr, a.status);
          if (!ok) break;
          gr ^= 1u << vs;
          clear_unseen(pc.u, j, vs, c, warp - nw, 4 - nw);
        }
        if (++vs == NS) { vs = 0; vr ^= 1; }
      }
    }
  }

  // ---- teardown ----
  tc_fence_before();
  __syncthreads();
  if (warp == 5) {
    __syncwarp();
    tmem_dealloc(tb, TMEM_COLS);
  }
}

// Merge of a unit's pieces: M = max m, L = sum l 2^(m - M), o = sum o 2^(m - M) / L, lse = ln2 (M + log2 L).  WPR warps
// per (sequence, token, head), D / 32 columns per lane, up to eight pieces in flight per warp; with several warps each
// takes every WPR-th group of eight and the partial results meet in shared memory.
template <int D, int WPR>
__global__ void __launch_bounds__(WPR == 1 ? 128 : WPR * 32) cowa_decode_tile_merge_kernel(const __grid_constant__ TileArgs a,
                                                                                         __nv_bfloat16* o, float* lse) {
  constexpr int V = D / 32, U = 8;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int r = WPR == 1 ? blockIdx.x * 4 + warp : blockIdx.x;
  if (r >= a.B * a.Nq * a.Hq) return;
  const int h = r % a.Hq, bt = r / a.Hq, t = bt % a.Nq, b = bt / a.Nq;
  const int tile = t / a.tpt, row = (t - tile * a.tpt) * a.G + h % a.G;
  const int u = (b * a.Hkv + h / a.G) * a.ntiles + tile;
  Unit x;
  unit_of(a, u, length_of(a, u), x);  // reads the lengths, which the tile kernel does not write: complete before that one began (grid_wait)
  grid_enter();      // the row states are complete and visible
  const int2 info = x.nt > 0 ? a.ws_unit[u] : make_int2(0, 0);  // no visible key: 0 / 0
  const size_t first = (size_t)(info.x + u) * a.rows + row;  // piece i lies a.rows rows further
  const int S = info.y;
  const float* po = a.ws_o + first * D + lane * V;
  float mx = -INFINITY, L = 0.f, acc[V];
#pragma unroll
  for (int i = 0; i < V; ++i) acc[i] = 0.f;
  for (int s0 = WPR == 1 ? 0 : warp * U; s0 < S; s0 += U * WPR) {
    // states and O of up to eight pieces in one round trip; the running maximum moves between such groups
    const float2 ml = lane < U && s0 + lane < S ? a.ws_ml[first + (size_t)(s0 + lane) * a.rows] : make_float2(-INFINITY, 0.f);
    float v[U][V];
#pragma unroll
    for (int k = 0; k < U; ++k) {
      const float* src = po + (size_t)(s0 + k) * a.rows * D;
      if constexpr (V == 4) {
        const float4 y = s0 + k < S ? *reinterpret_cast<const float4*>(src) : make_float4(0.f, 0.f, 0.f, 0.f);
        v[k][0] = y.x; v[k][1] = y.y; v[k][2] = y.z; v[k][3] = y.w;
      } else {
        const float2 y = s0 + k < S ? *reinterpret_cast<const float2*>(src) : make_float2(0.f, 0.f);
        v[k][0] = y.x; v[k][1] = y.y;
      }
    }
    float m = ml.x;
#pragma unroll
    for (int k = 4; k > 0; k >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, k));
    m = fmaxf(__shfl_sync(0xffffffffu, m, 0), mx);
    const float old = mx == -INFINITY ? 0.f : exp2f(mx - m), w = ml.x == -INFINITY ? 0.f : exp2f(ml.x - m);
    mx = m;
    float l = ml.y * w;
#pragma unroll
    for (int k = 4; k > 0; k >>= 1) l += __shfl_xor_sync(0xffffffffu, l, k);
    L = L * old + __shfl_sync(0xffffffffu, l, 0);
#pragma unroll
    for (int i = 0; i < V; ++i) acc[i] *= old;
#pragma unroll
    for (int k = 0; k < U; ++k) {
      const float wk = __shfl_sync(0xffffffffu, w, k);
#pragma unroll
      for (int i = 0; i < V; ++i) acc[i] = fmaf(v[k][i], wk, acc[i]);
    }
  }
  if constexpr (WPR > 1) {
    __shared__ float s_acc[WPR][D], s_m[WPR], s_l[WPR];
#pragma unroll
    for (int i = 0; i < V; ++i) s_acc[warp][lane * V + i] = acc[i];
    if (lane == 0) { s_m[warp] = mx; s_l[warp] = L; }
    __syncthreads();
    if (warp > 0) return;
    mx = s_m[0];
#pragma unroll
    for (int k = 1; k < WPR; ++k) mx = fmaxf(mx, s_m[k]);
    L = 0.f;
#pragma unroll
    for (int i = 0; i < V; ++i) acc[i] = 0.f;
#pragma unroll
    for (int k = 0; k < WPR; ++k) {
      const float w = s_m[k] == -INFINITY ? 0.f : exp2f(s_m[k] - mx);
      L = fmaf(s_l[k], w, L);
#pragma unroll
      for (int i = 0; i < V; ++i) acc[i] = fmaf(s_acc[k][lane * V + i], w, acc[i]);
    }
  }
  uint32_t pk[V / 2];
#pragma unroll
  for (int i = 0; i < V; i += 2) pk[i / 2] = pack_bf16(acc[i] / L, acc[i + 1] / L);
  __nv_bfloat16* dst = o + (size_t)r * D + lane * V;
  if constexpr (V == 4) *reinterpret_cast<uint2*>(dst) = make_uint2(pk[0], pk[1]);
  else *reinterpret_cast<uint32_t*>(dst) = pk[0];
  if (lse && lane == 0) lse[r] = 0.6931471805599453f * (mx + log2f(L));
}

// Shape of a call: row tiles, units, blocks and the workspace they need.
struct TilePlan {
  int tpt, ntiles, rows, blocks;
  long long units, steps;  // steps: of the longest possible list
  size_t bytes;
};

TilePlan plan_of(int B, int Nq, int Tmax, int Hq, int Hkv, int D, const cowa_params_t* p) {
  TilePlan t;
  const int G = Hq / Hkv;
  t.tpt = std::min(BQ / G, Nq);
  t.ntiles = (Nq + t.tpt - 1) / t.tpt;
  t.rows = t.tpt * G;
  t.units = (long long)B * Hkv * t.ntiles;
  // one wave of two blocks per SM, fewer when the longest possible list leaves a block less than two steps
  const int hg = p->hkv_global > 0 ? p->hkv_global : Hkv;
  long long vis = Tmax;
  if (!p->full_attn) {
    const long long shared = (long long)p->sink + p->local, band = (std::max((long long)Tmax - shared, 0ll) + hg - 1) / hg;
    vis = std::min<long long>(vis, shared + band + 3 * (BK + t.tpt));
  }
  t.steps = (vis + BK - 1) / BK * t.units;
  t.blocks = (int)std::max(1ll, std::min<long long>(2ll * cowa::sm_count(), (t.steps + 1) / 2));
  t.bytes = (size_t)(t.blocks + t.units) * t.rows * (D + 2) * sizeof(float) + (size_t)t.units * sizeof(int2);
  return t;
}

template <int D>
int launch_tile(const void* q, const void* kc, const void* vc, void* o, float* lse, int Tmax, const cowa_params_t* p,
                TileArgs& a, const TilePlan& t, void* ws, cudaStream_t st) {
  a.ws_o = static_cast<float*>(ws);
  a.ws_ml = reinterpret_cast<float2*>(a.ws_o + (size_t)(t.blocks + t.units) * t.rows * D);
  a.ws_unit = reinterpret_cast<int2*>(a.ws_ml + (size_t)(t.blocks + t.units) * t.rows);
  CUtensorMap mq, mk, mv;
  int rc;
  CowaStrides sq, sk;
  sq.t = D; sq.h = (long long)a.Hq * D; sq.b = (long long)a.Nq * a.Hq * D;  // q [B, Nq, Hq, D]: rows are heads, then tokens
  if ((rc = cowa::make_tensor_map(&mq, q, cowa::MapType::BF16, D, a.Hq, a.Nq, a.B, sq, 64, a.G, true, a.tpt))) return rc;
  const int rows = a.block_table ? a.page_size : Tmax;
  sk.t = D; sk.h = (long long)rows * D; sk.b = (long long)a.Hkv * rows * D;
  const int nb = a.block_table ? 0x7FFFFFFF : a.B;  // the pool's page count is not part of the call
  if ((rc = cowa::make_tensor_map(&mk, kc, cowa::MapType::BF16, D, rows, a.Hkv, nb, sk, 64, a.box))) return rc;
  if ((rc = cowa::make_tensor_map(&mv, vc, cowa::MapType::BF16, D, rows, a.Hkv, nb, sk, 64, a.box))) return rc;
  const bool few = t.rows <= 32;
  const auto kernel = few ? cowa_decode_tile_kernel<D, 32, 3> : cowa_decode_tile_kernel<D, 128, 2>;
  const int smem = few ? TileSmem<D, 32, 3>::kBytes : TileSmem<D, 128, 2>::kBytes;
  COWA_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
  COWA_CUDA_TRY(cowa::launch_chained(kernel, dim3((unsigned)t.blocks), kThreads, smem, st, mq, mk, mv, a));
  // one warp per row while a unit has a few pieces on average, eight warps when it has many (one long sequence)
  const bool many = t.blocks > 16 * t.units;
  const int nrows = a.B * a.Nq * a.Hq;
  const auto merge = many ? cowa_decode_tile_merge_kernel<D, 8> : cowa_decode_tile_merge_kernel<D, 1>;
  COWA_CUDA_TRY(cowa::launch_chained(merge, dim3((unsigned)(many ? nrows : (nrows + 3) / 4)), many ? 256 : 128, 0, st, a,
                                     static_cast<__nv_bfloat16*>(o), lse));
  return COWA_OK;
}

int decode_ext(const void* q, const void* kc, const void* vc, const int32_t* block_table, const int32_t* lens, void* o,
               float* lse, int B, int Nq, int Tmax, int page_size, int max_pages, int Hq, int Hkv, int D,
               const cowa_params_t* p, void* workspace, size_t workspace_bytes, void* stream) {
  int rc = cowa::decode_validate(q, kc, vc, lens, o, B, Tmax, Hq, Hkv, D, p);
  if (rc != COWA_OK) return rc;
  if (Nq <= 0 || Nq > 64 || !workspace) return COWA_ERR_INVALID_ARG;
  if (cowa::any_stride_set(p)) return COWA_ERR_UNSUPPORTED;
  if (!cowa::aligned16(workspace)) return COWA_ERR_MISALIGNED;
  const TilePlan t = plan_of(B, Nq, Tmax, Hq, Hkv, D, p);
  // units, the list of all their steps (t.steps leaves out partial tiles) and the merged rows are counted in 32 bits
  if (t.steps + 3 * t.units > 0x7FFFFFFFll || (long long)B * Nq * Hq > 0x7FFFFFFFll) return COWA_ERR_UNSUPPORTED;
  if (workspace_bytes < t.bytes) return COWA_ERR_WORKSPACE_TOO_SMALL;
  TileArgs a;
  a.lens = lens; a.block_table = block_table;
  a.status = cowa::device_status_word();
  if (!a.status) return COWA_ERR_CUDA;
  a.B = B; a.Nq = Nq; a.Hq = Hq; a.Hkv = Hkv; a.G = Hq / Hkv;
  a.tpt = t.tpt; a.ntiles = t.ntiles; a.rows = t.rows; a.units = (int)t.units;
  a.page_size = page_size; a.max_pages = max_pages;
  a.box = !block_table ? BK : page_size % 64 == 0 ? 64 : page_size % 32 == 0 ? 32 : 16;
  a.sink = p->sink; a.local = p->local;
  a.hkv_global = p->hkv_global > 0 ? p->hkv_global : Hkv;
  a.hkv_offset = p->hkv_offset; a.full_attn = p->full_attn;
  a.scale_log2 = p->softmax_scale * 1.4426950408889634f;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  return D == 128 ? launch_tile<128>(q, kc, vc, o, lse, Tmax, p, a, t, workspace, st)
                  : launch_tile<64>(q, kc, vc, o, lse, Tmax, p, a, t, workspace, st);
}

}  // namespace

extern "C" {

size_t cowa_decode_multi_workspace_bytes(int B, int Nq, int Tmax, int Hq, int Hkv, int D, const cowa_params_t* p) {
  if (!p || B <= 0 || Nq <= 0 || Tmax <= 0 || Hq <= 0 || Hkv <= 0 || Hq % Hkv != 0 || (D != 64 && D != 128)) return 0;
  if (Hq / Hkv > BQ) return 0;  // a group that does not fit a row tile (the calls take groups of up to 8)
  return plan_of(B, Nq, Tmax, Hq, Hkv, D, p).bytes;
}

int cowa_decode_multi(const void* q, const void* kcache, const void* vcache, const int32_t* lens, void* o,
                      float* lse, int B, int Nq, int Tmax, int Hq, int Hkv, int D, const cowa_params_t* p,
                      void* workspace, size_t workspace_bytes, void* stream) {
  return decode_ext(q, kcache, vcache, nullptr, lens, o, lse, B, Nq, Tmax, 0, 0, Hq, Hkv, D, p, workspace,
                    workspace_bytes, stream);
}

int cowa_decode_paged(const void* q, const void* kpages, const void* vpages, const int32_t* block_table,
                      const int32_t* lens, void* o, float* lse, int B, int Nq, int max_pages, int page_size,
                      int Hq, int Hkv, int D, const cowa_params_t* p, void* workspace, size_t workspace_bytes,
                      void* stream) {
  if (!block_table || max_pages <= 0 || page_size <= 0 || page_size % 16 != 0) return COWA_ERR_INVALID_ARG;
  if ((long long)max_pages * page_size > 0x7FFFFFFFll) return COWA_ERR_UNSUPPORTED;
  return decode_ext(q, kpages, vpages, block_table, lens, o, lse, B, Nq, max_pages * page_size, page_size, max_pages,
                    Hq, Hkv, D, p, workspace, workspace_bytes, stream);
}

}  // extern "C"
