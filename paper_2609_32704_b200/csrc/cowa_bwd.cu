// CoWindow Attention backward (Algorithm 2) for sm_100a.
//
// Three launches on the caller's stream, four when some KV tiles are shared:
//   1. preprocess   -Delta = -rowsum(O * dO) (Algorithm 2 line 13) and -LSE * log2(e), fp32 row vectors
//                   padded to a multiple of 64 rows (padding: -inf, so that P = 0 there);
//                   its threads also zero the fp32 dQ accumulator.
//   2. main kernel  a work item per (batch, KV head, 128-row KV tile), KV-stationary as in
//                   Algorithm 2, looping over the G QO heads of the group and over the 64-row QO
//                   tiles of I_h(j) (analytic scheduler, ascending).  A step takes two entries of that list, one
//                   head's after the other's, not necessarily neighbours (with 128-row tiles instead up to a
//                   tenth more rows were visited: windows of 300 and 466 keys).  Per step five tcgen05 MMAs:
//                     S^T  = K Q^T            (TMEM, 128 kv x 128 q)
//                     dP^T = V dO^T           (TMEM)
//                     dV  += P^T dO           (P^T as the TMEM operand)
//                     dK  += dS^T Q           (dS^T as the TMEM operand)
//                     dQ^T = K^T dS^T         (dS^T from shared memory; 128 d x 128 q in TMEM)
//                   dK and dV stay in TMEM for the whole loop, all G heads included, so they need no
//                   atomics (Algorithm 2 line 17 needs them only because it gives each QO head its
//                   own program).  dQ^T is drained by a separate warpgroup through shared memory and
//                   added to the fp32 accumulator with bulk add-reductions (Algorithm 2 line 15).
//                   Warp roles: scheduling / TMA producer / MMA issuer / two compute warpgroups (P, dS; each takes 64
//                   of the 128 query columns of every step) / dQ drain warpgroup, connected by mbarriers.
//                   What bounds it: shared memory.  Of a step's ~3920 clocks the products' operands take
//                   2048 (128 bytes a clock), the Q and dO loads 512, dS^T 256, the dQ staging 1024 written
//                   and read; the tensor pipe needs 2560, the exponentials 1024.  With steps of 64 queries
//                   K and V were read twice as often (2816), and a row constant per column and thread came
//                   out of shared memory as a broadcast (1024 more): 32K, 32 heads 7.83 -> 6.92 M cycles.  The
//                   512 columns of TMEM hold S^T, dP^T, dK, dV; P^T and dS^T take the outer halves of S^T
//                   and dP^T, dQ^T the 128 columns between them, so that the next S^T and dP^T only wait
//                   until dQ^T is in registers.  Per step n the MMAs run in the order
//                     dK(n-1) | dQ^T(n-1) | dP^T(n)   beside the exponentials of step n
//                     dV(n)   | S^T(n+1)              beside dS^T(n)
//                   At D = 128 S^T(n+1) is issued 1000 clocks later than dV(n) allows, when the second half of dQ^T has
//                   left its columns, behind the staging of the first (all 128 columns in registers at once: four copies
//                   of the staging code, 9 to 30 % slower; rotated through one copy: spills).  At D = 64 dQ^T has columns of
//                   its own, and the lanes that M = 128 leaves over hold it a second time, so that four warps
//                   drain it instead of two: a step of 3420 clocks waited 500 for dP^T and 450 for S^T(n+1).  us: 35584
//                   tokens, 32 heads 3433 -> 3190; 3840 x 4, 16 heads, reproducible 347 -> 296; 11120 x 2, 4 heads 252 -> 230.
//                   A second buffer for dO, which dP^T waited 250 clocks of the remaining 2835 for: 3280 -> 3155, 298 -> 291,
//                   234 -> 229.  What is left there is the chain of the compute warps; exponentials on the FMA pipe (one pair
//                   in eight or four) change nothing.
//                   Items are ordered sink tiles first (they meet every query tile), then
//                   head by head with ascending KV tile, so that the blocks in flight sweep the same
//                   dQ rows at nearly the same time and the reductions hit in L2.
//                   A block takes over further items (cluster launch control): between two blocks on an SM 2.5 us
//                   passed, and a block's first product came 1.4 us, its last store 5 us (D = 128) behind them; now Q and
//                   V of the next item arrive while the last products of this one run, K once dQ^T has read this
//                   one's, and its first S^T is computed while dK and dV leave through the buffers of dS^T and dO
//                   (straight from registers, 16 bytes of 32 rows at a time, they hold up the drain).  us, forward and
//                   backward: 2 x 8K 1004 -> 983, 20001 tokens 797 -> 766, 32K 7345 -> 7250, 24 documents 1564 -> 1546.
//   3. convert      dQ accumulator (already scaled) -> bf16.
// Two variations of the main kernel's work split:
//   - shared tiles: a tile's steps are cut into contiguous parts, an item each (few tiles, sink tiles that would
//     be the critical path, the last wave); each item writes fp32 partial dK, dV to its own slot and a
//     fourth kernel adds the slots in order (BwdPlan).
//   - VARLEN: packed batch [H, total, D]; the scheduling warp finds (sequence, KV tile) by a warp scan of the offsets,
//     windows follow from the sequence's own length, the accumulator and the row vectors use a row space
//     in which every sequence is padded to 64 rows, and a sequence's last, partial KV tile is stored row
//     by row (cowa_bwd_varlen and its own preprocess / convert kernels).
#include <cuda_bf16.h>

#include <algorithm>

#include "cowa_common.h"
#include "cowa_ptx.cuh"
#include "cowa_tma.h"

using namespace cowa_ptx;

namespace {

constexpr int BKV = 128;  // KV rows per block (MMA M)
constexpr int BQT = 128;  // QO rows per step (MMA N of S^T / dP^T): two tiles
constexpr int BQS = 64;   // rows of a QO tile, unit of the padded row space and of the plan's step counts
constexpr int NST = 2;    // Q stages (Q(n) is read again by dK(n) after S^T(n+1))
template <int D>
constexpr int NDO = D == 64 ? 2 : 1;  // dO stages: all that there is room for
constexpr int kNoTile = 0x7FFFFF00;  // in place of a step's second tile: no query of it sees anything
constexpr int kFewTiles = 296;  // up to so many tiles a batched call's plan is a table
constexpr float kDqFixedOne = 262144.f;  // 2^18: one unit of dQ in the fixed-point accumulation mode

struct BwdArgs {
  const float* lse2;   // [B*Hq, Tpad]  -LSE * log2(e)   (both negated: the packed adds have no operand negation)
  const float* delta;  // [B*Hq, Tpad]  -Delta
  float* dq_acc;       // fp32 [B*Hq, Tpad / 64, D / 32, 16, 32, 4]: 64 rows, 32 d, then four rows of one d (a drain warp's tile)
  unsigned int* status;
  int B, Nq, Nk, Hq, Hkv, G, Tpad;
  int sink_tiles;      // KV tiles per head that hold sink columns (launched first)
  // The KV tiles in launch order: sink tiles, body, tail.  A tile of class c is shared by cls_parts[c] blocks, each with
  // a contiguous part of the tile's steps (QO heads x QO tiles); a shared tile's blocks leave fp32 partial dK, dV.
  int cls_tiles[3], cls_parts[3];
  // Instead, where `few` is set: the items of one batch element are numbered tile after tile, KV tiles ascending, heads within
  // them, batch elements within the numbers; tile e = KV tile * Hkv + KV head has the numbers first[e] .. first[e + 1] - 1.
  int few;             // tiles of one batch element
  uint16_t first[kFewTiles + 1], shared[kFewTiles];  // shared: the tiles with several
  int single;          // the grid fits the device: a block has one item
  int dq_fixed;        // 1: dQ partial sums travel as 32-bit fixed point (order-independent addition)
  float* dkv_part;     // fp32 partial dK, dV [blocks of shared tiles, 2, BKV, D], summed by a kernel of their own
  // packed (variable-length) batches only: tensors are [H, total, D], sequence b owns rows cu[b] .. cu[b+1]
  const int* cu;       // [B+1] device
  __nv_bfloat16* dk;   // raw outputs for a sequence's last, partial KV tile and for tiles that no query sees
  __nv_bfloat16* dv;
  CowaStrides sdk, sdv;  // ... (packed batches: contiguous)
  int total, tiles_bound;  // rows of the packed tensors; grid tiles per KV head (upper bound of the real count)
  int sink, local, hkv_global, hkv_offset, full_attn, explicit_windows;
  float scale, scale_log2;
  CowaHeadWindows wins;
};

template <int D>
struct BwdSmem {
  static constexpr int kKV = BKV * D * 2;      // K or V tile
  static constexpr int kQ = BQT * D * 2;       // Q or dO tile of a step
  static constexpr int kDS = BKV * BQS * 2;    // dS^T of half a step (bf16)
  static constexpr int oK = 0, oV = kKV, oQ = 2 * kKV, oDO = oQ + NST * kQ, oDS = oDO + NDO<D> * kQ;
  static constexpr int oVec = oDS + 2 * kDS;   // per stage: 128 floats lse2, 128 floats delta
  static constexpr int oDQ = oVec + NST * 1024;  // dQ staging: per drain warp two tiles of 32 query rows x 32 d, fp32
  static constexpr int oBar = oDQ + 8 * 4096;
  static constexpr int oItem = oBar + 352;     // two work items
  static constexpr int oNext = oItem + 192;    // the next item's number, as the hardware answers
  static constexpr int kBytes = oNext + 16;    // 231984 B at D = 128 (limit 232448)
};

__device__ __forceinline__ void bulk_load_1d(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_u32(dst)),
               "l"(src), "r"(bytes), "r"(smem_u32(bar))
               : "memory");
}

// Tile number q of class c: sink tiles of every head first (they meet every query tile of their sequence and are the
// longest), then head-major with ascending KV tile (consecutive blocks share dQ rows, which then stay in L2).  Packed
// batches: the same sequence by sequence, longest first; whole warps only; false when there is no such tile (the count is an upper bound).
struct TileAt {
  int hk, b, j, nts, pbase;
};
// Packed batches: offsets that step back make sequences overlap, and their padded rows may outgrow the row space; such a
// sequence has no tiles here, the preprocess kernel reports it.  (With the report in this kernel it spilled, 332 bytes.)
__device__ __forceinline__ bool fits(const BwdArgs& a, const TileAt& x) {
  return (unsigned)x.pbase <= (unsigned)(a.Tpad - (a.cu[x.b + 1] - a.cu[x.b]));
}
template <bool VARLEN>
__device__ __forceinline__ bool locate_tile(const BwdArgs& a, int c, int q, TileAt& x) {
  const int nsk = a.sink_tiles, nhead = a.B * a.Hkv;
  x.pbase = 0;
  if (c == 0) {
    x.j = q / nhead; q %= nhead;
    x.hk = q % a.Hkv; x.b = q / a.Hkv;
    if constexpr (VARLEN) {
      varlen_seq_info(a.cu, x.b, BKV, BQS, &x.nts, &x.pbase);
      return x.j < x.nts && fits(a, x);  // else the sequence is shorter than its sink
    }
    return true;
  }
  if (c == 2) q += a.cls_tiles[1];
  if constexpr (VARLEN) {
    if (a.B <= kLongestFirst) {
      if (!varlen_locate_longest(a.cu, a.cu, a.B, q, BKV, a.Hkv, nsk, &x.b, &x.j, &x.nts)) return false;
      const int n = x.nts - nsk;
      x.hk = x.j / n; x.j = nsk + x.j % n;
      varlen_seq_info(a.cu, x.b, BKV, BQS, &x.nts, &x.pbase);
      return fits(a, x);
    }
    x.hk = q / a.tiles_bound;
    return varlen_locate(a.cu, a.B, q % a.tiles_bound, BKV, BQS, &x.b, &x.j, &x.nts, &x.pbase, nsk) && fits(a, x);
  }
  const int nrest = (a.Nk + BKV - 1) / BKV - nsk;
  x.j = nsk + q % nrest; q /= nrest;
  x.hk = q % a.Hkv; x.b = q / a.Hkv;
  return true;
}

// named barriers: one 128-thread warpgroup; all of the block, where the TMA warp does not wait
__device__ __forceinline__ void all_arrive() { asm volatile("bar.arrive 3, 512;" ::: "memory"); }
__device__ __forceinline__ void all_sync() { asm volatile("bar.sync 3, 512;" ::: "memory"); }
__device__ __forceinline__ void wg_sync(int id) { asm volatile("bar.sync %0, 128;" ::"r"(id) : "memory"); }

// One work item: a KV tile, or a part of its steps, as the scheduling warp publishes it for the others.
struct BwdItem {
  CowaWin w;
  int off, Nq, Nk;
  int steps;     // -1: no more items
  int k0, hk, b, rbase;
  float* part;   // where the partial dK, dV of a shared tile go, else nullptr
  // the TMA warp's: I_h(j), QO tiles per head and of this item, head of the group and position in I_h(j) of the first
  CowaRange rg[2];
  int cnt, tiles, g, t_in, pbase;
};
static_assert(sizeof(BwdItem) <= 96, "slot of a published item");
constexpr int kItemReaders = 14;  // warps that read it: TMA 1, MMA 1, compute 8, drain 4

template <int D, bool VARLEN>
__global__ void __launch_bounds__(512, 1)
cowa_bwd_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                const __grid_constant__ CUtensorMap tmV, const __grid_constant__ CUtensorMap tmdO,
                const __grid_constant__ CUtensorMap tmdK, const __grid_constant__ CUtensorMap tmdV,
                const __grid_constant__ CUtensorMap tmQ2, const __grid_constant__ CUtensorMap tmdO2,  // boxes of 128 rows
                const __grid_constant__ BwdArgs a) {
  using SM = BwdSmem<D>;
  constexpr int NSLAB = D / 64;
  constexpr int SLAB_KV = BKV * 128;  // bytes of one 64-wide slab of a 128-row tile
  constexpr int SLAB_Q = BQT * 128;   // ... of a Q or dO tile
  // TMEM columns
  constexpr uint32_t cS = 0, cDP = 128, cDK = 256, cDV = cDK + D, TMEM_COLS = 512;
  // P^T over the first half of S^T, dS^T over the second of dP^T, dQ^T between; at D = 64 there are columns left for it
  constexpr bool OWN_DQ = D == 64;
  constexpr uint32_t cDS = cDP + 64, cDQ = OWN_DQ ? 384 : cS + 64;
  constexpr uint32_t ID_ST = idesc_bf16(128, BQT, 0, 0);   // S^T, dP^T
  constexpr uint32_t ID_ACC = idesc_bf16(128, D, 0, 1);    // dV, dK (B = dO / Q, MN-major)
  constexpr uint32_t ID_DQ = idesc_bf16(128, BQT, 1, 1);   // dQ^T (A = K^T, B = dS^T, both MN-major)

  extern __shared__ __align__(1024) uint8_t smem[];
  uint8_t* sK = smem + SM::oK;
  uint8_t* sV = smem + SM::oV;
  uint8_t* sQ = smem + SM::oQ;
  uint8_t* sDO = smem + SM::oDO;
  uint8_t* sDS = smem + SM::oDS;
  float* sVec = reinterpret_cast<float*>(smem + SM::oVec);
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + SM::oBar);
  uint64_t* bar_k = bars + 0;
  uint64_t* bar_v = bars + 6;
  uint64_t* bar_q_full = bars + 1;    // [2] Q, LSE, Delta of a step have landed
  uint64_t* bar_q_empty = bars + 3;   // [2] ... are consumed
  uint64_t* bar_o_full = bars + 37;   // [NDO] dO ...
  uint64_t* bar_o_empty = bars + 39;  // [NDO]
  uint64_t* bar_s_full = bars + 7;    // S^T is in TMEM
  uint64_t* bar_s_read = bars + 8;    // count 256: S^T is in registers
  uint64_t* bar_p_ready = bars + 9;   // count 256: P^T written over the first half of S^T
  uint64_t* bar_dp_full = bars + 10;  // dP^T is in TMEM
  uint64_t* bar_ds_ready = bars + 11; // count 256: dS^T in TMEM (over the second half of dP^T) and shared memory
  uint64_t* bar_dq_full = bars + 12;  // dQ^T is in TMEM
  uint64_t* bar_dq_free = bars + 13;  // [2] count 128: ... has left the columns of dP^T, of S^T
  uint64_t* bar_done = bars + 15;
  uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(bars + 16);
  // What the roles would otherwise each hold or compute (registers: nothing spills in the batched form)
  int2* step_info = reinterpret_cast<int2*>(bars + 18);        // [2] by stage: first queries of the step's tiles; bit 0: no pair is masked, bit 1: rows past the sequence's end
  longlong2* dq_at = reinterpret_cast<longlong2*>(bars + 20);  // [4] by step: first elements of its tiles' dQ rows, -1: no second tile
  uint64_t* bar_i_full = bars + 29;   // [2] a work item has been published
  uint64_t* bar_i_empty = bars + 31;  // [2] count kItemReaders: it has been read
  uint64_t* bar_next = bars + 33;     // the next item's number is here
  uint64_t* bar_dk_out = bars + 34;   // dK of an item has left the buffer of dS^T
  uint64_t* bar_dv_out = bars + 35;   // dV ... of dO
  uint64_t* bar_ask = bars + 36;      // it is time to ask for the next item
  auto item_at = [&](uint32_t ni) { return reinterpret_cast<BwdItem*>(smem + SM::oItem + (ni & 1) * 96); };

  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);  // warp-uniform by construction (helps the compiler)

  if (tid == 0) {
    mbar_init(bar_k, 1); mbar_init(bar_v, 1);
    for (int s = 0; s < 2; ++s) {
      mbar_init(bar_q_full + s, 1); mbar_init(bar_q_empty + s, 1);
      mbar_init(bar_dq_free + s, 128);
      mbar_init(bar_o_full + s, 1); mbar_init(bar_o_empty + s, 1);
      mbar_init(bar_i_full + s, 1); mbar_init(bar_i_empty + s, kItemReaders);
    }
    mbar_init(bar_dq_full, 1);
    mbar_init(bar_s_full, 1); mbar_init(bar_s_read, 256); mbar_init(bar_p_ready, 256);
    mbar_init(bar_dp_full, 1); mbar_init(bar_ds_ready, 256);
    mbar_init(bar_done, 1); mbar_init(bar_next, 1); mbar_init(bar_dk_out, 1); mbar_init(bar_dv_out, 1); mbar_init(bar_ask, 1);
    fence_mbar_init();
  }
  if (tid == 32) { prefetch_tmap(&tmQ2); prefetch_tmap(&tmdO2); prefetch_tmap(&tmK); prefetch_tmap(&tmV); }
  __syncthreads();
  // What needs nothing of the kernel before this one is done ahead of the wait for it: this, and the first item's geometry (not so
  // the TMEM allocation, see cowa_fwd_kernel; the first loads do not wait for that).  A grid that is not started as a whole cannot
  // let the next kernel in early.
  auto enter = [&]() {
    if (a.single) grid_enter();
    else grid_wait();
  };
  if (warp == 0 || warp == 2) {
    all_arrive();
    if (VARLEN || warp == 0) enter();
  } else {
    enter();
    if (warp == 1) {
      __syncwarp();
      tmem_alloc(tmem_holder, TMEM_COLS);
      tmem_relinquish();
    }
    tc_fence_before();
    all_sync();
    tc_fence_after();
  }
  constexpr uint32_t tmem_base = 0;  // the allocation is all of TMEM

  // dO of step c: its stage, and the parity of its turn there
  auto o_stage = [](int c) { return NDO<D> == 2 ? c & 1 : 0; };
  auto o_turn = [](int c) { return (uint32_t)(NDO<D> == 2 ? c >> 1 : c) & 1; };

  bool ok = true;
  // Item number ni of this block has been published (its words stay until item_done); its steps, -1 when there are no more items.
  auto next_item = [&](uint32_t ni) -> int {
    ok = mbar_wait(bar_i_full + (ni & 1), (ni >> 1) & 1, a.status);
    return ok ? static_cast<const volatile int*>(&item_at(ni)->steps)[0] : -1;
  };
  auto item_done = [&](uint32_t ni) {
    __syncwarp();
    if (lane == 0) mbar_arrive(bar_i_empty + (ni & 1));
  };

  // Register budget per role: 128 per thread at launch (512 threads), 80 + 2 * 152 + 128 = 4 * 128 moved to where the work
  // is.  Each setmaxnreg sits at the top of its own branch so that the code below it is compiled for that budget.
  if (warp < 4) {
    setmaxnreg_dec<80>();
    if (warp == 2) {
      // ================= scheduling: takes over items and works out their geometry, one ahead of the others =================
      // (In the TMA warp this came between two items' loads: 1.6 us, 3.5 us in packed batches.)
      const bool lead = elect_one();
      int idx = blockIdx.x;
      uint32_t asked = 0;
      auto next_index = [&]() {
        if (a.single) return -1;
        if (lead) {
          mbar_expect_tx(bar_next, 16);
          clc_request(smem + SM::oNext, bar_next);
        }
        ok = mbar_wait(bar_next, asked & 1, a.status);
        ++asked;
        if (!ok) return -1;
        const int x = __shfl_sync(0xFFFFFFFFu, clc_block(smem + SM::oNext), 0);
        fence_proxy_async_smem();  // read before the next answer is written
        __syncwarp();
        return x;
      };
      for (uint32_t ni = 0; ok;) {
        BwdItem it;
        it.steps = -1;
        if (idx >= 0) {
          int parts = 1, part = 0, slot = idx;  // slot: of this item's partial dK, dV when the tile is shared
          TileAt at;
          bool found = true;
          if (!VARLEN && a.few > 0) {
            const int q = idx / a.B;
            int e = 0, hi = a.few - 1;  // the last tile with first[e] <= q
            while (e < hi) {
              const int mid = (e + hi + 1) >> 1;
              if (a.first[mid] <= q) e = mid;
              else hi = mid - 1;
            }
            parts = a.first[e + 1] - a.first[e]; part = q - a.first[e];
            at.b = idx - q * a.B; at.hk = e % a.Hkv; at.j = e / a.Hkv; at.pbase = 0;
          } else {
            int cls = 0, q = idx;
            slot = 0;
            while (cls < 2 && q >= a.cls_tiles[cls] * a.cls_parts[cls]) {
              q -= a.cls_tiles[cls] * a.cls_parts[cls];
              if (a.cls_parts[cls] > 1) slot += a.cls_tiles[cls] * a.cls_parts[cls];
              ++cls;
            }
            parts = a.cls_parts[cls]; part = q % parts;
            slot += q;
            found = locate_tile<VARLEN>(a, cls, q / parts, at);
          }
          // Sequence geometry.  Packed batches: N_q = N_k = the sequence's length, rows start at cu[b]; the fp32
          // dQ accumulator and the LSE / Delta vectors are laid out with every sequence padded to 64 rows (pbase).
          it.Nq = a.Nq; it.Nk = a.Nk; it.rbase = 0;
          if (found) it.w = a.wins.w[at.hk];
          if (VARLEN && found) {
            it.rbase = a.cu[at.b];
            it.Nq = it.Nk = a.cu[at.b + 1] - it.rbase;
            if (it.rbase < 0 || it.rbase + it.Nk > a.total) {  // malformed offsets: report, touch nothing
              if (lead) atomicOr(a.status, (unsigned)COWA_DEV_BAD_SEQLENS);
              found = false;
            }
            if (a.full_attn) { it.w.s = 0; it.w.n = it.Nk; it.w.g = 0; it.w.l = 0; }
            else if (!a.explicit_windows) it.w = cowa_default_window(it.Nk, a.hkv_global, a.hkv_offset + at.hk, a.sink, a.local);
          }
          if (!found) {  // (packed batches: the count of items is an upper bound)
            idx = next_index();
            continue;
          }
          it.hk = at.hk; it.b = at.b; it.pbase = at.pbase; it.off = it.Nk - it.Nq; it.k0 = at.j * BKV;
          cowa_bwd_ranges(it.w, it.k0, min(it.k0 + BKV, it.Nk) - 1, it.off, it.Nq, BQS, it.rg);
          it.cnt = cowa_range_len(it.rg[0]) + cowa_range_len(it.rg[1]);
          const int n0 = it.cnt * a.G * part / parts;        // (the host checks that these products fit)
          it.tiles = it.cnt * a.G * (part + 1) / parts - n0;
          it.steps = (it.tiles + 1) >> 1;
          it.g = it.cnt > 0 ? n0 / it.cnt : 0; it.t_in = n0 - it.g * it.cnt;
          it.part = parts > 1 ? a.dkv_part + (size_t)slot * 2 * (BKV * D) : nullptr;
        }
        if (ni >= 2) ok = mbar_wait(bar_i_empty + (ni & 1), ((ni >> 1) & 1) ^ 1, a.status);
        if (!ok) break;
        if (lead) {
          *item_at(ni) = it;
          mbar_arrive(bar_i_full + (ni & 1));
        }
        __syncwarp();
        if (it.steps < 0) break;
        if (!a.single) ok = mbar_wait(bar_ask, ni & 1, a.status, cowa_bwd_item_clocks(it.steps));  // nearly all of the item
        ++ni;
        if (ok) idx = next_index();
      }
    } else if (warp == 0) {
      // ================= TMA producer =================
      const bool lead = elect_one();
      int c = 0;        // steps so far, all items together
      uint32_t kc = 0;  // items with steps so far
      for (uint32_t ni = 0; ok; ++ni) {
        const int N = next_item(ni);
        if (N < 0) break;
        const volatile BwdItem* const it = item_at(ni);
        CowaWin w;
        w.s = it->w.s; w.n = it->w.n; w.g = it->w.g; w.l = it->w.l;
        const int off = it->off, Nq = it->Nq, Nk = it->Nk, k0 = it->k0, hk = it->hk, b = it->b, rbase = it->rbase;
        const int cnt = it->cnt, tiles = it->tiles, pbase = it->pbase;
        int g = it->g, t_in = it->t_in;  // kept incrementally
        CowaRange rg[2];
        rg[0].lo = it->rg[0].lo; rg[0].hi = it->rg[0].hi; rg[1].lo = it->rg[1].lo; rg[1].hi = it->rg[1].hi;
        item_done(ni);
        auto ask = [&]() {
          if (lead && !a.single) mbar_arrive(bar_ask);
        };
        const int bt = VARLEN ? 0 : b;                   // batch coordinate of the tensor maps
        const int hq0 = hk * a.G;                        // first QO head of the group
        const int bhq0 = (VARLEN ? 0 : b * a.Hq) + hq0;  // ... as a row of lse2 / delta / dq_acc
        auto load_kv = [&](uint8_t* tile, const CUtensorMap* tm, uint64_t* bar) {
          if (!lead) return;
          mbar_expect_tx(bar, SM::kKV);
          for (int s = 0; s < NSLAB; ++s) tma_load_4d(tile + s * SLAB_KV, tm, bar, s * 64, rbase + k0, hk, bt);
        };
        if (c == 0 && N > 0) load_kv(sK, &tmK, bar_k);  // S^T of the first step waits for K and Q only
        const int ask_at = max(N - 4, 0);               // some microseconds before the next item is needed
        if (N == 0) ask();
        for (int n = 0; n < N; ++n, ++c) {
          const int st = c & 1;
          if (n == ask_at) ask();
          int q0[2], gh[2];
          q0[0] = cowa_bwd_tile_at(rg, t_in) * BQS; gh[0] = g;
          if (++t_in == cnt) { t_in = 0; ++g; }
          const bool two = 2 * n + 1 < tiles;  // else the first tile again, every pair of it masked
          q0[1] = two ? cowa_bwd_tile_at(rg, t_in) * BQS : q0[0]; gh[1] = two ? g : gh[0];
          if (two && ++t_in == cnt) { t_in = 0; ++g; }
          // neighbours of one head, as nearly always, come in one piece
          const int pieces = two && gh[1] == gh[0] && q0[1] == q0[0] + BQS ? 1 : 2;
          auto load_rows = [&](uint8_t* tile, const CUtensorMap* tm, const CUtensorMap* tm2, uint64_t* bar) {
            for (int x = 0; x < pieces; ++x)
              for (int s = 0; s < NSLAB; ++s)
                tma_load_4d(tile + s * SLAB_Q + x * (SLAB_Q / 2), pieces == 1 ? tm2 : tm, bar, s * 64, rbase + q0[x], hq0 + gh[x], bt);
          };
          if (c >= 2) ok = mbar_wait(bar_q_empty + st, ((c >> 1) & 1) ^ 1, a.status);
          if (!ok) break;
          if (lead) {
            auto info = [&](int x) {
              return q0[x] + (cowa_tile_full(w, q0[x], BQS, k0, BKV, off, Nq, Nk) ? 1 : 0) + (q0[x] + BQS > Nq ? 2 : 0);
            };
            step_info[st] = make_int2(info(0), two ? info(1) : kNoTile);
            auto rows = [&](int x) -> size_t { return (size_t)(bhq0 + gh[x]) * a.Tpad + pbase + q0[x]; };  // in lse2, delta, dq_acc
            dq_at[c & 3] = make_longlong2((long long)rows(0) * D, two ? (long long)rows(1) * D : -1ll);
            mbar_expect_tx(bar_q_full + st, SM::kQ + 2 * BQT * 4);
            load_rows(sQ + st * SM::kQ, &tmQ, &tmQ2, bar_q_full + st);
            for (int x = 0; x < pieces; ++x) {
              bulk_load_1d(sVec + st * 256 + x * BQS, a.lse2 + rows(x), BQT * 4 / pieces, bar_q_full + st);
              bulk_load_1d(sVec + st * 256 + 128 + x * BQS, a.delta + rows(x), BQT * 4 / pieces, bar_q_full + st);
            }
          }
          if (n == 0) {  // V over that of the item before once its last dP^T has been computed, K once dQ^T has
            if (c > 0) ok = mbar_wait(bar_dp_full, (c - 1) & 1, a.status);
            if (!ok) break;
            load_kv(sV, &tmV, bar_v);
          }
          // (dV of the item before has left the buffer of dO: behind dO's last product)
          if (n == 0 && c > 0) ok = mbar_wait(bar_dv_out, (kc - 1) & 1, a.status);
          else if (c >= NDO<D>) ok = mbar_wait(bar_o_empty + o_stage(c), o_turn(c) ^ 1, a.status);
          if (!ok) break;
          if (lead) {
            mbar_expect_tx(bar_o_full + o_stage(c), SM::kQ);
            load_rows(sDO + o_stage(c) * SM::kQ, &tmdO, &tmdO2, bar_o_full + o_stage(c));
          }
          if (n == 0 && c > 0) {
            ok = mbar_wait(bar_dq_full, (c - 1) & 1, a.status);
            if (!ok) break;
            load_kv(sK, &tmK, bar_k);
          }
          __syncwarp();
        }
        if (!ok) break;
        if (N > 0) ++kc;
      }
    } else if (warp == 1) {
      // ================= MMA issuer =================
      // The whole warp runs this loop (uniform control flow, so that descriptors and counters stay in
      // uniform registers); only the elected lane executes the tcgen05 instructions.  Everything that
      // can be computed once is: descriptor of every operand base, stage and parity bookkeeping is
      // incremental.
      {
        const bool lead = elect_one();
        const uint32_t tb = tmem_base;
        // Descriptors: a byte offset o inside a tile is added as o >> 4 to the address field (bits 0-13);
        // no tile crosses the field's range, so the 64-bit add never carries out of it.
        const uint64_t dK_k = smem_desc_sw128(smem_u32(sK), 16, 1024);                       // K, K-major (A of S^T)
        const uint64_t dV_k = smem_desc_sw128(smem_u32(sV), 16, 1024);                       // V, K-major (A of dP^T)
        const uint64_t dK_mn = smem_desc_sw128(smem_u32(sK), D == 128 ? SLAB_KV : 0, 1024);  // K^T, MN-major (A of dQ^T)
        const uint64_t dQ_k0 = smem_desc_sw128(smem_u32(sQ), 16, 1024);        // Q of stage 0, K-major (B of S^T)
        const uint64_t dO_k0 = smem_desc_sw128(smem_u32(sDO), 16, 1024);       // dO of stage 0, K-major (B of dP^T)
        const uint64_t dQ_mn0 = smem_desc_sw128(smem_u32(sQ), SLAB_Q, 1024);   // Q, MN-major (B of dK)
        const uint64_t dO_mn0 = smem_desc_sw128(smem_u32(sDO), SLAB_Q, 1024);  // dO, MN-major (B of dV)
        const uint64_t dDS = smem_desc_sw128(smem_u32(sDS), SM::kDS, 1024);    // dS^T, MN-major (B of dQ^T)
        constexpr uint32_t kQ16 = SM::kQ >> 4;

        auto gemm_st = [&](uint32_t d_col, uint64_t dA, uint64_t dB) {  // [128 x 128] = A[128 x D] B[128 x D]^T
          if (lead) {
#pragma unroll
            for (int kk = 0; kk < D / 16; ++kk)
              mma_ss(tb + d_col, dA + (((kk / 4) * SLAB_KV + (kk % 4) * 32) >> 4),
                     dB + (((kk / 4) * SLAB_Q + (kk % 4) * 32) >> 4), ID_ST, kk > 0);
          }
        };
        auto gemm_acc = [&](uint32_t d_col, uint32_t a_col, uint64_t dB, uint32_t acc_first) {  // [128 x D] += A(TMEM) B
          if (lead) {
#pragma unroll
            for (int kk = 0; kk < BQT / 16; ++kk)  // 32-query blocks 0, 2 from one warpgroup's columns, 1, 3 from the other's
              mma_ts(tb + d_col, tb + a_col + ((kk >> 1) & 1) * 32 + (kk >> 2) * 16 + (kk & 1) * 8, dB + ((kk * 2048) >> 4), ID_ACC, kk > 0 ? 1u : acc_first);
          }
        };
        auto gemm_dq = [&]() {  // dQ^T[D x 128] = K^T dS^T
          if (lead) {
#pragma unroll
            for (int kk = 0; kk < BKV / 16; ++kk)
              mma_ss(tb + cDQ, dK_mn + ((kk * 2048) >> 4), dDS + ((kk * 2048) >> 4), ID_DQ, kk > 0);
          }
        };
        auto commit = [&](uint64_t* bar) {
          if (lead) mma_commit(bar);
        };

        const BwdItem* item = nullptr;
        // Packed batches: rows of a tile that lie past the end of the sequence belong to the next one.  Every
        // product they enter is multiplied by an exact zero, but 0 x (Inf or NaN) would still poison this
        // sequence, so they are cleared in shared memory (whole 128-byte rows, by this warp) before use.
        auto clear_rows = [&](uint8_t* tile, int first, int rows, int slab_bytes) {
          const int nchunk = (rows - first) * 8;  // 16-byte chunks per slab
          for (int s_ = 0; s_ < NSLAB; ++s_)
            for (int c_ = lane; c_ < nchunk; c_ += 32)
              *reinterpret_cast<uint4*>(tile + s_ * slab_bytes + first * 128 + c_ * 16) = make_uint4(0u, 0u, 0u, 0u);
        };
        auto clear_tail = [&](uint8_t* tile, int stage) {  // Q or dO of the step whose Q is in this stage
          if constexpr (VARLEN) {
            const int2 q0_ = step_info[stage];
            if (!((q0_.x | q0_.y) & 2)) return;
            const int nq = static_cast<const volatile int*>(&item->Nq)[0];
#pragma unroll 1
            for (int x = 0; x < 2; ++x) {
              const int q = x && q0_.y != kNoTile ? q0_.y : q0_.x;  // (without a second tile the first lies there again)
              if (q & 2) clear_rows(tile + x * (SLAB_Q / 2), nq - (q & ~63), BQS, SLAB_Q);
            }
            fence_proxy_async_smem();
            __syncwarp();
          }
        };
        auto clear_kv_tail = [&](uint8_t* tile) {
          if constexpr (VARLEN) {
            const int left = static_cast<const volatile int*>(&item->Nk)[0] - static_cast<const volatile int*>(&item->k0)[0];
            if (left >= BKV) return;
            clear_rows(tile, left, BKV, SLAB_KV);
            fence_proxy_async_smem();
            __syncwarp();
          }
        };
        int c = 0;        // steps so far: stage, parities
        uint32_t kc = 0;  // items with steps so far
        // Step n of an item.  What it waits for of the step before it holds across items, too.
        auto body = [&](int n, int N) {
          const int st = c & 1;
          const uint32_t par = c & 1;
          if (n > 0) {
            ok = mbar_wait(bar_ds_ready, par ^ 1, a.status);
            if (!ok) return;
            tc_fence_after();
            gemm_acc(cDK, cDS, dQ_mn0 + (st ^ 1) * kQ16, n > 1 ? 1u : 0u);
            commit(bar_q_empty + (st ^ 1));
            // dQ^T's columns: S^T of this step is in registers; or those of its own, once the dQ^T before it has left them
            if (!OWN_DQ) ok = mbar_wait(bar_s_read, par, a.status);
            else if (c > 1) ok = mbar_wait(bar_dq_free, par, a.status);
            if (!ok) return;
            tc_fence_after();
            gemm_dq();
            commit(bar_dq_full);
          }
          ok = mbar_wait(bar_o_full + o_stage(c), o_turn(c), a.status);
          if (!OWN_DQ && ok && c > 0) ok = mbar_wait(bar_dq_free, par ^ 1, a.status);
          if (!ok) return;
          if (n == 0) {
            ok = mbar_wait(bar_v, kc & 1, a.status);
            if (!ok) return;
            clear_kv_tail(sV);
          }
          clear_tail(sDO + o_stage(c) * SM::kQ, st);
          tc_fence_after();
          gemm_st(cDP, dV_k, dO_k0 + o_stage(c) * kQ16);
          commit(bar_dp_full);
          ok = mbar_wait(bar_p_ready, par, a.status);
          if (!ok) return;
          tc_fence_after();
          gemm_acc(cDV, cS, dO_mn0 + o_stage(c) * kQ16, n > 0 ? 1u : 0u);
          commit(bar_o_empty + o_stage(c));
          if (n + 1 < N) {
            ok = mbar_wait(bar_q_full + (st ^ 1), ((c + 1) >> 1) & 1, a.status);
            if (!OWN_DQ && ok && c > 0) ok = mbar_wait(bar_dq_free + 1, par ^ 1, a.status);
            if (!ok) return;
            clear_tail(sQ + (st ^ 1) * SM::kQ, st ^ 1);
            tc_fence_after();
            gemm_st(cS, dK_k, dQ_k0 + (st ^ 1) * kQ16);
            commit(bar_s_full);
          }
        };
        for (uint32_t ni = 0; ok; ++ni) {
          const int N = next_item(ni);
          if (N < 0) break;
          item = item_at(ni);
          if (N > 0) {
            ok = mbar_wait(bar_k, kc & 1, a.status);
            if (!ok) break;
            clear_kv_tail(sK);
            ok = mbar_wait(bar_q_full + (c & 1), (c >> 1) & 1, a.status);
            if (!OWN_DQ && ok && c > 0) ok = mbar_wait(bar_dq_free + 1, (c - 1) & 1, a.status);
            if (!ok) break;
            clear_tail(sQ + (c & 1) * SM::kQ, c & 1);
            tc_fence_after();
            gemm_st(cS, dK_k, dQ_k0 + (c & 1) * kQ16);
            commit(bar_s_full);
#pragma unroll 1
            for (int n = 0; n < N && ok; ++n, ++c) body(n, N);
            if (!ok) break;
            ok = mbar_wait(bar_ds_ready, (c - 1) & 1, a.status);
            if (ok && c > 1) ok = mbar_wait(bar_dq_free + (OWN_DQ ? 0 : 1), c & 1, a.status);
            if (!ok) break;
            tc_fence_after();
            gemm_dq();  // K may go now
            commit(bar_dq_full);
            gemm_acc(cDK, cDS, dQ_mn0 + ((c - 1) & 1) * kQ16, N > 1 ? 1u : 0u);
            commit(bar_q_empty + ((c - 1) & 1));
            commit(bar_done);
            ++kc;
          }
          item_done(ni);
        }
      }
    }
  } else if (warp < 12) {
    setmaxnreg_inc<152>();
    {
      // ======== two compute warpgroups: P^T and dS^T of two blocks of 32 queries each.  A warpgroup only writes into
      // columns that it has read: P^T (bf16 pairs) into its first block of S^T, dS^T into its second of dP^T.
      const int wg = (warp - 4) >> 2;  // queries [32 wg, 32 wg + 32) of both halves of every step
      // A thread holds the fragments of the 16-lane TMEM accesses: keys row0 + {0, 8, 16, 24}, query pairs 8 j + 2 (lane % 4)
      // of every 32-query block: eight row constants a block instead of 32 broadcast ones.
      const int lane4 = lane >> 2, pair = (lane & 3) * 2;
      const uint32_t t_lane = tmem_base + ((uint32_t)((warp & 3) * 32) << 16);
      const uint32_t ds_st = smem_u32(sDS) + ((warp & 3) * 32 + (lane & 15)) * 128;  // this lane's row for stmatrix
      const uint32_t ds_ch = wg * 4 + (lane >> 4);                                   // ... and 16-byte chunk
      const float2 sc2 = make_float2(a.scale_log2, a.scale_log2);
      int c = 0;        // steps so far: stage, parities
      uint32_t kc = 0;  // items with steps so far
      for (uint32_t ni = 0; ok; ++ni) {
      const int N = next_item(ni);
      if (N < 0) break;
      // queries that see this lane's key: [near_lo, near_hi] and [far_lo, far_hi]
      int near_lo = 0, near_hi = -1, far_lo = 0, far_hi = -1;
      {
        const volatile BwdItem* it = item_at(ni);
        const int kcol = it->k0 + (warp & 3) * 32 + lane;
        const long long kpos = (long long)kcol - it->off, qend = it->Nq - 1, far = kpos + it->w.n + it->w.g;
        if (kcol < it->Nk) {
          near_lo = (int)max(min(kpos, qend + 1), 0ll);
          near_hi = (int)max(kcol < it->w.s ? qend : min(kpos + it->w.n - 1, qend), -1ll);
          far_lo = (int)max(min(far, qend + 1), 0ll);
          far_hi = (int)max(it->w.l > 0 ? min(far + it->w.l - 1, qend) : -1ll, -1ll);
        }
      }
      for (int n = 0; n < N && ok; ++n, ++c) {
        const int st = c & 1;
        const uint32_t par = c & 1;
        const uint32_t sbuf = t_lane + cS + wg * 32, dpbuf = t_lane + cDP + wg * 32;
        const float2* nlse2 = reinterpret_cast<const float2*>(sVec + st * 256 + wg * 32 + pair);  // -LSE log2(e), then -Delta
        ok = mbar_wait(bar_q_full + st, (c >> 1) & 1, a.status);
        float2 rc[8];  // row constants, read ahead of the wait for the product: shared memory is busy with its operands
#pragma unroll
        for (int j = 0; j < 8; ++j) rc[j] = nlse2[(j >> 2) * 32 + (j & 3) * 4];
        const int2 info = step_info[st];
        const bool full = info.x & info.y & 1;
        uint32_t mk[2], all[2] = {0xFFFFFFFFu, 0xFFFFFFFFu}, seen[2] = {0xFFFFFFFFu, 0xFFFFFFFFu};
        if (!full) {
#pragma unroll
          for (int cb = 0; cb < 2; ++cb) {
            const int base = ((cb ? info.y : info.x) & ~63) + wg * 32;
            mk[cb] = interval_bits(near_lo, near_hi, base) | interval_bits(far_lo, far_hi, base);
            all[cb] = __ballot_sync(0xffffffffu, mk[cb] == 0xFFFFFFFFu);
            seen[cb] = __ballot_sync(0xffffffffu, mk[cb] != 0u);
          }
        }
        ok = ok && mbar_wait(bar_s_full, par, a.status);
        if (!ok) break;
        tc_fence_after();
        float p[2][2][16];  // [query block][16-key half]
#pragma unroll
        for (int cb = 1; cb >= 0; --cb)
#pragma unroll
          for (int h = 0; h < 2; ++h)
            tmem_ld_frag(sbuf + cb * 64 + ((uint32_t)(h * 16) << 16), p[cb][h]);
        tmem_wait_ld();
        tc_fence_before();
        if constexpr (!OWN_DQ) mbar_arrive(bar_s_read);
#pragma unroll
        for (int cb = 0; cb < 2; ++cb) {
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            float* x = p[cb][h];
            // of a boundary step only the 16 keys x 32 queries that the boundary crosses are masked, and those beyond it zeroed
            if ((seen[cb] >> (h * 16)) & 0xFFFFu) {
#pragma unroll
              for (int e = 0; e < 16; e += 2) {
                const float2 y = fma2(make_float2(x[e], x[e + 1]), sc2, rc[cb * 4 + e / 4]);
                x[e] = ex2(y.x);
                x[e + 1] = ex2(y.y);
              }
              if (((all[cb] >> (h * 16)) & 0xFFFFu) != 0xFFFFu) {
                const uint32_t m0 = __shfl_sync(0xffffffffu, mk[cb], h * 16 + lane4) >> pair;
                const uint32_t m1 = __shfl_sync(0xffffffffu, mk[cb], h * 16 + 8 + lane4) >> pair;
#pragma unroll
                for (int e = 0; e < 16; ++e)
                  if (!((((e & 2) ? m1 : m0) >> ((e >> 2) * 8 + (e & 1))) & 1u)) x[e] = 0.f;
              }
            } else {
#pragma unroll
              for (int e = 0; e < 16; ++e) x[e] = 0.f;
            }
            uint32_t pk[8];
#pragma unroll
            for (int e = 0; e < 16; e += 2) pk[e / 2] = pack_bf16(x[e], x[e + 1]);
            tmem_st_frag(sbuf + cb * 16 + ((uint32_t)(h * 16) << 16), pk);  // P^T: 32 queries as 16 bf16 pairs
          }
        }
        tmem_wait_st();
        tc_fence_before();
        mbar_arrive(bar_p_ready);
#pragma unroll
        for (int j = 0; j < 8; ++j) rc[j] = nlse2[64 + (j >> 2) * 32 + (j & 3) * 4];

        ok = mbar_wait(bar_dp_full, par, a.status);
        if (ok && n == 0 && kc > 0) ok = mbar_wait(bar_dk_out, (kc - 1) & 1, a.status);
        if (!ok) break;
        tc_fence_after();
#pragma unroll
        for (int cb = 1; cb >= 0; --cb) {  // (dS^T goes where the second block was)
          float dr[2][16];
#pragma unroll
          for (int h = 0; h < 2; ++h) tmem_ld_frag(dpbuf + cb * 64 + ((uint32_t)(h * 16) << 16), dr[h]);
          tmem_wait_ld();
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            uint32_t dsp[8];
#pragma unroll
            for (int e = 0; e < 16; e += 2) {
              const float2 y = mul2(make_float2(p[cb][h][e], p[cb][h][e + 1]), add2(make_float2(dr[h][e], dr[h][e + 1]), rc[cb * 4 + e / 4]));
              dsp[e / 2] = pack_bf16(y.x, y.y);
            }
            tmem_st_frag(dpbuf + 64 + cb * 16 + ((uint32_t)(h * 16) << 16), dsp);
            // dS^T also to shared memory (a key's row = 128 B = 8 chunks, 128B swizzle) for the dQ^T product, whose last
            // reading of the tile is complete: it was issued ahead of dP^T
#pragma unroll
            for (int j = 0; j < 4; j += 2)
              stmatrix4(ds_st + cb * SM::kDS + h * 2048 + (((ds_ch + j) ^ (lane & 7)) << 4), dsp + 2 * j);
          }
        }
        tmem_wait_st();
        tc_fence_before();
        fence_proxy_async_smem();
        mbar_arrive(bar_ds_ready);
      }
      if (!ok) break;
      // dK (first warpgroup) and dV (second, while the last dQ^T and dK are still being computed).  K, V and Q of the next item
      // arrive meanwhile.
      const bool is_dk = wg == 0;
      const int r = (warp & 3) * 32 + lane;
      if (N > 0) {
        ok = is_dk ? mbar_wait(bar_done, kc & 1, a.status) : mbar_wait(bar_o_empty + o_stage(c - 1), o_turn(c - 1), a.status);
        if (!ok) break;
        ++kc;
      }
      tc_fence_after();
      const uint32_t acc = t_lane + (is_dk ? cDK : cDV);
      const float mul = is_dk ? a.scale : 1.f;
      const BwdItem* it = item_at(ni);
      if (float* const part = it->part) {
        // A shared tile: this item's part goes out in fp32, one slot per item; a kernel of its own adds the slots in order.  A slot
        // holds 16 bytes of every row after the other, so that a warp's store is one range of 512 bytes.
        float4* const d4 = reinterpret_cast<float4*>(part + (is_dk ? 0 : BKV * D)) + r;
#pragma unroll
        for (int q = 0; q < D / 32; ++q) {
          uint32_t ov[32];
          if (N > 0) {
            tmem_ld32(acc + q * 32, ov);
            tmem_wait_ld();
          } else {
#pragma unroll
            for (int e = 0; e < 32; ++e) ov[e] = 0u;
          }
#pragma unroll
          for (int e = 0; e < 8; ++e)
            d4[(q * 8 + e) * BKV] = make_float4(__uint_as_float(ov[e * 4]) * mul, __uint_as_float(ov[e * 4 + 1]) * mul,
                                                __uint_as_float(ov[e * 4 + 2]) * mul, __uint_as_float(ov[e * 4 + 3]) * mul);
        }
        __syncwarp();
        if (N > 0 && r == 0) mbar_arrive(is_dk ? bar_dk_out : bar_dv_out);  // (nothing staged)
      } else {
        const int left = it->Nk - it->k0;  // rows of this tile
        // Through shared memory, but for the last, partial KV tile of a packed sequence, whose other rows belong to the next one, and
        // for a tile that no query sees: the two barriers count items with steps, as a role that has none could get two ahead.
        const bool staged = N > 0 && !(VARLEN && left < BKV);
        const CowaStrides sd = is_dk ? a.sdk : a.sdv;
        __nv_bfloat16* const dst = (is_dk ? a.dk : a.dv) + (VARLEN ? 0 : (size_t)it->b * sd.b) + (size_t)it->hk * sd.h +
                                   (size_t)(it->rbase + it->k0 + r) * sd.t;
        uint8_t* const sOut = (is_dk ? sDS : sDO + o_stage(c - 1) * SM::kQ) + r * 128;
#pragma unroll
        for (int q = 0; q < D / 32; ++q) {
          uint32_t ov[32];
          if (N > 0) {
            tmem_ld32(acc + q * 32, ov);
            tmem_wait_ld();
          } else {
#pragma unroll
            for (int e = 0; e < 32; ++e) ov[e] = 0u;
          }
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            uint4 v;
            v.x = pack_bf16(__uint_as_float(ov[e * 8 + 0]) * mul, __uint_as_float(ov[e * 8 + 1]) * mul);
            v.y = pack_bf16(__uint_as_float(ov[e * 8 + 2]) * mul, __uint_as_float(ov[e * 8 + 3]) * mul);
            v.z = pack_bf16(__uint_as_float(ov[e * 8 + 4]) * mul, __uint_as_float(ov[e * 8 + 5]) * mul);
            v.w = pack_bf16(__uint_as_float(ov[e * 8 + 6]) * mul, __uint_as_float(ov[e * 8 + 7]) * mul);
            const int slab = q / 2, chunk = (q & 1) * 4 + e;
            if (staged) *reinterpret_cast<uint4*>(sOut + slab * SLAB_KV + ((chunk ^ (r & 7)) << 4)) = v;
            else if (r < left) *reinterpret_cast<uint4*>(dst + q * 32 + e * 8) = v;
          }
        }
        if (staged) {
          fence_proxy_async_smem();
          wg_sync(is_dk ? 1 : 2);
        }
        if (N > 0 && r == 0) {
          if (staged) {
            const int bt = VARLEN ? 0 : it->b;
            for (int s = 0; s < NSLAB; ++s)
              tma_store_4d(is_dk ? &tmdK : &tmdV, sOut + s * SLAB_KV, s * 64, it->rbase + it->k0, it->hk, bt);
            tma_commit_group();
            tma_wait_group_read<0>();
          }
          mbar_arrive(is_dk ? bar_dk_out : bar_dv_out);
        }
      }
      tc_fence_before();
      item_done(ni);
      }
    }
  } else {
    {
      // ======== dQ drain warpgroup: one d column of dQ^T per thread; TMEM -> shared -> bulk reduce-add ========
      float* sDQ = reinterpret_cast<float*>(smem + SM::oDQ) + (warp & 3) * 2048;
      const uint32_t t_lane = tmem_base + ((uint32_t)((warp & 3) * 32) << 16);
      // At D = 64 the lanes 64 to 127 hold the same as the first 64 (K^T is read twice as A): these two warps take half 0.
      const int d_part = warp & (D / 32 - 1);  // this warp's 32 d
      int c = 0;  // steps so far
      for (uint32_t ni = 0; ok; ++ni) {
      const int N = next_item(ni);
      if (N < 0) break;
      item_done(ni);
      for (int n = 0; n < N && ok; ++n, ++c) {
        ok = mbar_wait(bar_dq_full, c & 1, a.status);
        if (!ok) break;
        tc_fence_after();
        // 32 query rows of this warp's 32 d: staged in one of two tiles and added to the accumulator as one range
        const longlong2 at_ = dq_at[c & 3];
        auto add_rows = [&](const uint32_t (&v)[32], int half, int odd) {
          const long long at = half ? at_.y : at_.x;
          if (at < 0) return;
          float* stage = sDQ + odd * 1024;
          if (lane == 0) tma_wait_group_read<1>();  // the reduction issued from this tile before has read it
          __syncwarp();
          if (a.dq_fixed) {
            // Rounded to integers on the FMA and integer pipes (the conversion instruction runs at the rate of the
            // exponentials and competes with them): below 2^22, x + 1.5 * 2^23 has rint(x) in its low mantissa bits.  Larger
            // ones go in two parts, x = 2^16 h + l with h = rint(x / 2^16), |l| <= 2^15, both exact; shifting the first
            // sum by 16 drops its exponent.  Both give what __float2int_rn gives for the product x rounded to fp32 (in one
            // FMA with the addition it would not be rounded, and an element's bits would depend on its neighbours' size).
            const float2 fx2 = make_float2(a.scale * kDqFixedOne, a.scale * kDqFixedOne);
            auto c2 = [](float c_) { return make_float2(c_, c_); };
            float worst = 0.f;
#pragma unroll
            for (int c = 0; c < 32; c += 2)
              worst = max_nan(worst, max_nan(fabsf(__uint_as_float(v[c])), fabsf(__uint_as_float(v[c + 1]))));
            worst *= fabsf(fx2.x);
            if (__all_sync(0xffffffffu, worst < 4194303.f)) {
#pragma unroll
              for (int c = 0; c < 32; c += 4) {
                const float2 x = mul2(make_float2(__uint_as_float(v[c]), __uint_as_float(v[c + 1])), fx2);
                const float2 y = mul2(make_float2(__uint_as_float(v[c + 2]), __uint_as_float(v[c + 3])), fx2);
                auto low = [](float t) { return __float_as_int(__fadd_rn(t, 12582912.f)) - 0x4B400000; };  // (a packed addition is merged)
                *reinterpret_cast<int4*>(stage + c * 32 + lane * 4) = make_int4(low(x.x), low(x.y), low(y.x), low(y.y));
              }
            } else {
#pragma unroll
              for (int c = 0; c < 32; c += 4) {
                int o[4];
#pragma unroll
                for (int e = 0; e < 4; e += 2) {
                  const float2 x = mul2(make_float2(__uint_as_float(v[c + e]), __uint_as_float(v[c + e + 1])), fx2);
                  const float2 th = fma2(x, c2(1.f / 65536.f), c2(12582912.f));
                  const float2 l = fma2(add2(th, c2(-12582912.f)), c2(-65536.f), x);
                  const float2 tl = add2(l, c2(12582912.f));
                  o[e] = (__float_as_int(th.x) << 16) + (__float_as_int(tl.x) - 0x4B400000);
                  o[e + 1] = (__float_as_int(th.y) << 16) + (__float_as_int(tl.y) - 0x4B400000);
                }
                *reinterpret_cast<int4*>(stage + c * 32 + lane * 4) = make_int4(o[0], o[1], o[2], o[3]);
              }
              if (!(worst < 2147483520.f)) atomicOr(a.status, (unsigned)COWA_DEV_DQ_RANGE);  // would not fit 32 bits (or NaN)
            }
          } else {
#pragma unroll
            for (int c = 0; c < 32; c += 4)
              *reinterpret_cast<float4*>(stage + c * 32 + lane * 4) =
                  make_float4(__uint_as_float(v[c]) * a.scale, __uint_as_float(v[c + 1]) * a.scale,
                              __uint_as_float(v[c + 2]) * a.scale, __uint_as_float(v[c + 3]) * a.scale);
          }
          fence_proxy_async_smem();
          __syncwarp();
          if (lane == 0) {
            float* dst = a.dq_acc + at + d_part * (BQS * 32) + odd * 1024;
            if (a.dq_fixed) bulk_reduce_add_s32(dst, stage, 4096);
            else bulk_reduce_add_f32(dst, stage, 4096);
            tma_commit_group();
          }
        };
        // First the columns that dP^T waits for, then those of S^T.  One loop body, like the MMA warp's: the roles' loops
        // together outgrow the instruction cache (two and four copies: 32K 7660 us forward and backward, this 7410).
#pragma unroll 1
        for (int half = OWN_DQ ? (warp & 3) < 2 : 1, last = OWN_DQ ? half : 0; half >= last; --half) {
          uint32_t v0[32], v1[32];
          tmem_ld32(t_lane + cDQ + half * 64, v0);
          tmem_ld32(t_lane + cDQ + half * 64 + 32, v1);
          tmem_wait_ld();
          tc_fence_before();
          mbar_arrive(bar_dq_free + (OWN_DQ ? 0 : half ^ 1));
          add_rows(v0, half, 0);
          add_rows(v1, half, 1);
        }
      }
      }
      if (lane == 0) tma_wait_group_read<0>();
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    __syncwarp();
    tmem_dealloc(tmem_base, TMEM_COLS);
  }
}

// delta = -rowsum(O * dO), lse2 = -LSE * log2(e); rows in [T, Tpad) get lse2 = -inf, delta = 0.  The same threads zero
// the fp32 dQ accumulator (as a memset before it that was a pass of its own: 32K 190 us for both, 164 us so).
template <int D>
__global__ void cowa_bwd_preprocess_kernel(const __nv_bfloat16* o, const __nv_bfloat16* d_o, const float* lse, float* lse2,
                                           float* delta, float* acc, int T, int Tpad, long long BH, int H, CowaStrides so) {
  grid_enter();
  constexpr int TPR = D / 8;  // threads per row (16 bytes each)
  const long long gid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const long long row = gid / TPR;
  const int part = (int)(gid % TPR);
  if (row >= BH * Tpad) return;
  const long long bh = row / Tpad;
  const int t = (int)(row % Tpad);
  // All loads ahead of the first store: the compiler does not move them over it.
  uint4 x = make_uint4(0u, 0u, 0u, 0u), y = x;
  float l = -INFINITY, s = 0.f;
  if (t < T) {
    const size_t base = (size_t)(bh / H) * so.b + (size_t)(bh % H) * so.h + (size_t)t * so.t + part * 8;
    x = *reinterpret_cast<const uint4*>(o + base);
    y = *reinterpret_cast<const uint4*>(d_o + base);
    if (part == 0) l = lse[(size_t)bh * T + t] * -1.4426950408889634f;
  }
  float4* z = reinterpret_cast<float4*>(acc + (size_t)row * D + part * 8);
  z[0] = z[1] = make_float4(0.f, 0.f, 0.f, 0.f);
  const uint32_t xs[4] = {x.x, x.y, x.z, x.w}, ys[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    s = fmaf(__uint_as_float(xs[i] << 16), __uint_as_float(ys[i] << 16), s);
    s = fmaf(__uint_as_float(xs[i] & 0xffff0000u), __uint_as_float(ys[i] & 0xffff0000u), s);
  }
#pragma unroll
  for (int o_ = TPR / 2; o_ > 0; o_ >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o_);
  if (part == 0) {
    delta[row] = -s;
    lse2[row] = l;
  }
}

// Packed batches.  One block per (64-row chunk of the padded row space, QO head): -Delta and -LSE * log2(e)
// of the chunk's rows (padding rows: -inf, 0), read from the packed tensors.  Bound by memory: a thread clears its part of
// the accumulator before it knows where the rows lie, and has all its loads in flight together (24 documents of 40000
// tokens, 16 heads: one row a thread 142 us, this 102; 680 MB).
template <int D>
__global__ void __launch_bounds__(256)
cowa_bwd_preprocess_varlen_kernel(const __nv_bfloat16* o, const __nv_bfloat16* d_o, const float* lse, float* lse2, float* delta,
                                  float* acc, const int* cu, int B, int total, int Tpad, unsigned int* status) {
  grid_enter();
  constexpr int TPR = D / 8;                          // threads per row (16 bytes each)
  constexpr int ROWS = 256 / TPR, PASS = BQS / ROWS;  // rows at a time
  const int chunk = blockIdx.x, h = blockIdx.y;
  const int r0 = threadIdx.x / TPR, part = threadIdx.x % TPR;
  float4* z = reinterpret_cast<float4*>(acc + ((size_t)h * Tpad + (size_t)chunk * BQS) * D);
#pragma unroll
  for (int i = 0; i < BQS * D / 4 / 256; ++i) z[i * 256 + threadIdx.x] = make_float4(0.f, 0.f, 0.f, 0.f);
  int b, lc, nch, pb;
  if (chunk == 0 && h == 0 && threadIdx.x < 32 && varlen_locate(cu, B, Tpad / BQS, BQS, BQS, &b, &lc, &nch, &pb) &&
      threadIdx.x == 0)
    atomicOr(status, (unsigned)COWA_DEV_BAD_SEQLENS);  // more chunks than the row space holds: see fits
  const bool in = varlen_locate(cu, B, chunk, BQS, BQS, &b, &lc, &nch, &pb);
  const int rbase = in ? cu[b] : 0, first = in ? rbase + lc * BQS : 0;  // the chunk's first row among the packed ones
  const int rows = !in || rbase < 0 ? 0 : min(cu[b + 1], total) - first;
  uint4 x[PASS], y[PASS];
  float l[PASS];
#pragma unroll
  for (int i = 0; i < PASS; ++i) {
    const int r = r0 + i * ROWS;
    x[i] = y[i] = make_uint4(0u, 0u, 0u, 0u);
    l[i] = -INFINITY;
    if (r < rows) {
      const size_t row = (size_t)h * total + first + r;
      x[i] = *reinterpret_cast<const uint4*>(o + row * D + part * 8);
      y[i] = *reinterpret_cast<const uint4*>(d_o + row * D + part * 8);
      if (part == 0) l[i] = lse[row] * -1.4426950408889634f;
    }
  }
#pragma unroll
  for (int i = 0; i < PASS; ++i) {
    const uint32_t xs[4] = {x[i].x, x[i].y, x[i].z, x[i].w}, ys[4] = {y[i].x, y[i].y, y[i].z, y[i].w};
    float s = 0.f;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      s = fmaf(__uint_as_float(xs[e] << 16), __uint_as_float(ys[e] << 16), s);
      s = fmaf(__uint_as_float(xs[e] & 0xffff0000u), __uint_as_float(ys[e] & 0xffff0000u), s);
    }
#pragma unroll
    for (int o_ = TPR / 2; o_ > 0; o_ >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o_);
    if (part == 0) {
      const size_t row = (size_t)h * Tpad + (size_t)chunk * BQS + r0 + i * ROWS;  // chunks are laid out in order: pb == chunk * BQS
      delta[row] = -s;
      lse2[row] = l[i];
    }
  }
}

// The dQ accumulator to bf16: one 64-row chunk of the row space and one head a block, every row's 16-byte pieces of four
// rows and one d (see the drain); a thread takes four rows of two d, so that a warp reads 1 KB ranges and writes whole
// sectors.
template <int D, bool VARLEN>
__device__ __forceinline__ void convert_dq(const float* acc, __nv_bfloat16* dq, const int* cu, int B, int T, int Tpad, int fixed,
                                           const CowaStrides& sq, int H, unsigned int* status, int chunk, int bh) {
  int rows, first;  // rows of this chunk, and the first one's place among the rows of dq
  __nv_bfloat16* out;
  if constexpr (!VARLEN) {
    first = chunk * BQS;
    rows = T - first;
    out = dq + (size_t)(bh / H) * sq.b + (size_t)(bh % H) * sq.h;
  } else {
    int b, lc, nch, pb;
    if (!varlen_locate(cu, B, chunk, BQS, BQS, &b, &lc, &nch, &pb)) return;
    const int rbase = cu[b];
    first = rbase + lc * BQS;
    rows = rbase < 0 ? 0 : min(cu[b + 1], T) - first;
    out = dq + (size_t)bh * sq.h;
  }
  const float4* src = reinterpret_cast<const float4*>(acc + ((size_t)bh * Tpad + (size_t)chunk * BQS) * D);
#pragma unroll
  for (int i = 0; i < D / 32; ++i) {
    const int item = i * 256 + threadIdx.x, r = item / 16 % 16 * 4, d = item / 256 * 32 + item % 16 * 2;
    float4 x = src[item * 2], y = src[item * 2 + 1];
    if (fixed) {
      const float u = 1.f / kDqFixedOne;
      x = make_float4(__float_as_int(x.x) * u, __float_as_int(x.y) * u, __float_as_int(x.z) * u, __float_as_int(x.w) * u);
      y = make_float4(__float_as_int(y.x) * u, __float_as_int(y.y) * u, __float_as_int(y.z) * u, __float_as_int(y.w) * u);
      // half of the representable range: a total that wrapped around lands out here in most cases
      const float big = fmaxf(fmaxf(fmaxf(fabsf(x.x), fabsf(x.y)), fmaxf(fabsf(x.z), fabsf(x.w))),
                              fmaxf(fmaxf(fabsf(y.x), fabsf(y.y)), fmaxf(fabsf(y.z), fabsf(y.w))));
      if (big >= 4096.f) atomicOr(status, (unsigned)COWA_DEV_DQ_RANGE);
    }
    const uint32_t v[4] = {pack_bf16(x.x, y.x), pack_bf16(x.y, y.y), pack_bf16(x.z, y.z), pack_bf16(x.w, y.w)};
#pragma unroll
    for (int e = 0; e < 4; ++e)
      if (r + e < rows) *reinterpret_cast<uint32_t*>(out + (size_t)(first + r + e) * sq.t + d) = v[e];
  }
}

template <int D, bool VARLEN>
__global__ void __launch_bounds__(256)
cowa_bwd_convert_dq_kernel(const float* acc, __nv_bfloat16* dq, const int* cu, int B, int T, int Tpad, int H, int fixed,
                           CowaStrides sq, unsigned int* status) {
  grid_enter();
  const int nchunk = Tpad / BQS;
  convert_dq<D, VARLEN>(acc, dq, cu, B, T, Tpad, fixed, sq, H, status, blockIdx.x % nchunk, blockIdx.x / nchunk);
}

// Partial dK (m = 0) and dV (1) of the shared tiles, added in slot order, to bf16.
template <int D>
constexpr int kReduceBlocks = BKV * (D / 8) / 256;  // of a tile and m: a thread takes eight d of a row, a warp 32 rows (see the slots)
template <int D, bool VARLEN>
__device__ __forceinline__ void reduce_dkv(const BwdArgs& a, const CowaStrides& sk, const CowaStrides& sv, int block, int m) {
  const int i_ = block % kReduceBlocks<D> * 256 + threadIdx.x, r = i_ % BKV, part = i_ / BKV;
  int q = block / kReduceBlocks<D>, c = 0, slot = 0, parts, step = 1;  // the tile's slots: slot, slot + step, ...
  TileAt at;
  if (!VARLEN && a.few > 0) {
    const int e = a.shared[q / a.B];
    at.b = q % a.B; at.hk = e % a.Hkv; at.j = e / a.Hkv;
    parts = a.first[e + 1] - a.first[e];
    slot = a.first[e] * a.B + at.b; step = a.B;
  } else {
  for (; c < 2; ++c) {
    if (a.cls_parts[c] == 1) continue;
    if (q < a.cls_tiles[c]) break;
    q -= a.cls_tiles[c];
    slot += a.cls_tiles[c] * a.cls_parts[c];
  }
  parts = a.cls_parts[c];
  if (!locate_tile<VARLEN>(a, c, q, at)) return;
  slot += q * parts;
  }
  int Nk = a.Nk, rbase = 0;
  if constexpr (VARLEN) {
    rbase = a.cu[at.b];
    Nk = a.cu[at.b + 1] - rbase;
    if (rbase < 0 || rbase + Nk > a.total) return;
  }
  const int t = at.j * BKV + r;
  if (t >= Nk) return;
  const float* src = a.dkv_part + ((size_t)slot * 2 + m) * (BKV * D) + ((size_t)part * 2 * BKV + r) * 4;
  float4 x = make_float4(0.f, 0.f, 0.f, 0.f), y = x;
#pragma unroll 4
  for (int i = 0; i < parts; ++i) {
    const float4 u = *reinterpret_cast<const float4*>(src + (size_t)i * step * 2 * (BKV * D));
    const float4 v = *reinterpret_cast<const float4*>(src + (size_t)i * step * 2 * (BKV * D) + BKV * 4);
    x.x += u.x; x.y += u.y; x.z += u.z; x.w += u.w;
    y.x += v.x; y.y += v.y; y.z += v.z; y.w += v.w;
  }
  const size_t o = VARLEN ? ((size_t)at.hk * a.total + rbase + t) * D
                 : m == 0 ? (size_t)at.b * sk.b + (size_t)at.hk * sk.h + (size_t)t * sk.t
                          : (size_t)at.b * sv.b + (size_t)at.hk * sv.h + (size_t)t * sv.t;
  *reinterpret_cast<uint4*>((m == 0 ? a.dk : a.dv) + o + part * 8) =
      make_uint4(pack_bf16(x.x, x.y), pack_bf16(x.z, x.w), pack_bf16(y.x, y.y), pack_bf16(y.z, y.w));
}

template <int D, bool VARLEN>
__global__ void __launch_bounds__(256)
cowa_bwd_reduce_dkv_kernel(const __grid_constant__ BwdArgs a, CowaStrides sk, CowaStrides sv) {
  grid_enter();
  reduce_dkv<D, VARLEN>(a, sk, sv, blockIdx.x, blockIdx.y);
}

// Both in one launch, the sums first, where the accumulator is small: a kernel less in the chain (forward and
// backward of 1024 tokens, 4 heads, with the table of tiles 25.8 -> 23.0 us).  Long
// ones keep the conversion's occupancy (with the registers of the sums 137 instead of 112 us at 32K).
template <int D, bool VARLEN>
__global__ void __launch_bounds__(256)
cowa_bwd_finish_kernel(const __grid_constant__ BwdArgs a, CowaStrides sk, CowaStrides sv, int sums, __nv_bfloat16* dq, int T, CowaStrides sq) {
  grid_enter();
  const int i = blockIdx.x - sums, nchunk = a.Tpad / BQS;
  if (i < 0) reduce_dkv<D, VARLEN>(a, sk, sv, blockIdx.x >> 1, blockIdx.x & 1);
  else convert_dq<D, VARLEN>(a.dq_acc, dq, a.cu, a.B, T, a.Tpad, a.dq_fixed, sq, a.Hq, a.status, i % nchunk, i / nchunk);
}
constexpr int kFinishChunks = 2048;  // 64-row chunks of the accumulator, all heads together

// How the KV tiles are shared among blocks.  A tile whose block takes the whole GQA group keeps dK, dV in TMEM; a shared
// tile costs every block a prologue and 128 KB of fp32 partial sums (D = 128), so tiles are shared only where whole ones
// leave SMs idle (work and shares are counted in 64-row QO tiles here, half a step of the kernel each):
//   sink tiles, visited by every query tile, when one is longer than 3/4 of an SM's share of the work: thirds of a share;
//   all tiles when there are at most two per SM: fifths of a share, four QO tiles at least;
//   the last tile per SM when there are at most eight: quarters, so that the last wave ends together.
// These lines were measured with steps of one QO tile instead of two and have been left where they are; what a body tile's
// block costs with the longer steps is in choose_run, which takes fewer of the parts reserved here.
struct BwdPlan {
  int sink_tiles;  // per sequence and head
  int tiles[3], parts[3];  // parts: what the workspace has room for
  int run[3];              // what the blocks take
  // ... or, batched calls of few tiles (BwdArgs)
  int few = 0, few_shared = 0;
  long long few_blocks = 0;
  uint16_t first[kFewTiles + 1], shared[kFewTiles];
  long long slots() const {
    long long n = 0;
    for (int c = 0; c < 3; ++c)
      if (parts[c] > 1) n += (long long)tiles[c] * parts[c];
    return n;
  }
  long long blocks() const {
    if (few > 0) return few_blocks;
    long long n = 0;
    for (int c = 0; c < 3; ++c) n += (long long)tiles[c] * run[c];
    return n;
  }
  // How many of the parts of body tiles are worth a block: a block costs about four steps (128 queries each) besides its own
  // and 0.02 for its partial sums, and half a block is lost at the end.  Forward and backward, us, all parts / these: 821
  // tokens x 4 (2 KV heads) 113 / 107, 2048 tokens 103 / 99, 6000 tokens 165 / 145, 20001 tokens 785 / 766; 1024 tokens, less
  // than a block per SM, 31 with four parts and 36 with two.  Reproducible gradients take all parts: other groups of steps
  // would give dK and dV other bits (20001 tokens 782 / 803).
  void choose_run(double steps, bool reproducible) {
    for (int c = 0; c < 3; ++c) run[c] = parts[c];
    if (reproducible) return;
    const int sms = cowa::sm_count();
    double best = 0;
    for (int p = 1; p <= parts[1]; ++p) {
      const long long n = (long long)tiles[0] * parts[0] + (long long)tiles[1] * p + (long long)tiles[2] * parts[2];
      const double t = (4 + steps / p) * (std::max((double)n / sms, 1.0) + 0.5) + (p > 1 ? 0.02 * tiles[1] * p : 0);
      if (p == 1 || t < best) { best = t; run[1] = p; }
    }
  }

  // Few tiles: their blocks by length.  With the same number of parts for every tile the blocks of a causal batch have one to
  // fourteen steps, and the last SM ends at twice the average (821 tokens x 4, 16 heads: SMs end after 23 to 60 us).
  // Of shares an eighth apart the one that ends first, as far as can be told: an item costs about as much as five QO
  // tiles besides its own, a block five more, and its partial sums 0.04; with more items than SMs a part of one is lost at the end.  cnt: QO tiles
  // of each KV tile of one batch element.
  void share_out(const int* cnt, int n, int B, long long total, int longest) {
    const int sms = cowa::sm_count();
    const long long room = std::min<long long>(slots(), 65535ll * B);
    double best = 0;
    int share = 0;
    for (int x = std::max(longest, 4);; x = std::max(x * 7 / 8, 4)) {
      long long b = 0;
      for (int i = 0; i < n; ++i) b += std::max((cnt[i] + x - 1) / x, 1);
      b *= B;
      if (b > room) break;
      double t = 10 + x;
      if (b > sms) t = std::max(t, 5 + (total + 5. * b) / sms + 0.4 * (5 + x));
      if (b > (long long)n * B) t += 0.04 * b;
      if (share == 0 || t < best) { best = t; share = x; few_blocks = b; }
      if (x == 4) break;
    }
    if (share == 0) return;
    few = n;
    int at = 0;
    for (int i = 0; i < n; ++i) {
      const int parts = std::max((cnt[i] + share - 1) / share, 1);
      first[i] = (uint16_t)at;
      at += parts;
      if (parts > 1) shared[few_shared++] = (uint16_t)i;
    }
    first[n] = (uint16_t)at;
  }
};

// `rest` KV tiles behind the sink tiles, `avg` QO tiles each; share: an SM's QO tiles
void plan_rest(BwdPlan& pl, long long rest, double avg, double share) {
  const int sms = cowa::sm_count();
  pl.tiles[1] = (int)rest; pl.parts[1] = 1;
  pl.tiles[2] = 0; pl.parts[2] = 1;
  if (rest <= 2 * sms) {
    pl.parts[1] = std::max(1, std::min(16, (int)(avg / std::max(share / 5, 4.0) + 0.999)));
  } else if (rest <= 8ll * sms && avg >= 16) {
    pl.tiles[2] = sms;
    pl.tiles[1] -= pl.tiles[2];
    pl.parts[2] = avg >= 32 ? 4 : 2;
  }
}

BwdPlan bwd_plan(int B, int Nq, int Nk, int Hkv, int G, const CowaHeadWindows& hw, bool reproducible) {
  BwdPlan pl;
  const int nKV = (Nk + BKV - 1) / BKV, sms = cowa::sm_count();
  pl.sink_tiles = 0;
  for (int h = 0; h < Hkv; ++h) pl.sink_tiles = std::max(pl.sink_tiles, (std::min(hw.w[h].s, Nk) + BKV - 1) / BKV);
  long long total = 0, sinks = 0, longest = 0, longest_sink = 0, longest_rest = 0;
  int counts[kFewTiles];  // tile j of head h: [j * Hkv + h]
  // (A table's parts do not end with the heads: items side by side no longer sweep the same rows of Q and dQ, which is lost where
  // these outgrow L2: 31232 tokens, 8 heads 4850 / 4980 us with it.  It costs in long sequences already: us, without / with it,
  // local 2000: 8192 tokens, 8 heads of one KV head 220 / 277, 4087 tokens x 4 336 / 372.  So with it where sequences are short,
  // 2000 tokens x 4 154 / 122, 3000 x 3 175 / 147, or a class has a part well above an SM's share, 8000 tokens, 4 heads 152 / 93.)
  const bool few = (long long)nKV * Hkv * B <= std::min(2 * sms, kFewTiles) && (long long)B * Hkv * G * Nq <= 131072;
  for (int h = 0; h < Hkv; ++h)
    for (int j = 0; j < nKV; ++j) {
      CowaRange rg[2];
      const int k0 = j * BKV, k1 = std::min(k0 + BKV, Nk) - 1;
      cowa_bwd_ranges(hw.w[h], k0, k1, Nk - Nq, Nq, BQS, rg);
      const long long cnt = (long long)(cowa_range_len(rg[0]) + cowa_range_len(rg[1])) * G;
      total += cnt;
      if (few) counts[j * Hkv + h] = (int)cnt;
      longest = std::max(longest, cnt);
      if (j < pl.sink_tiles) { sinks += cnt; longest_sink = std::max(longest_sink, cnt); }
      else longest_rest = std::max(longest_rest, cnt);
    }
  total *= B; sinks *= B;
  const double share = (double)total / sms;
  const long long rest = (long long)B * Hkv * (nKV - pl.sink_tiles);
  pl.tiles[0] = B * Hkv * pl.sink_tiles;
  pl.parts[0] = longest_sink * 4 > 3 * share ? std::max(1, std::min(32, (int)(longest_sink / std::max(share / 3, 4.0) + 0.999))) : 1;
  plan_rest(pl, rest, rest > 0 ? (double)(total - sinks) / rest : 0.0, share);
  // Memory for partial sums: `heads` slots per tile, the smallest divisor of G that gives two waves of blocks and keeps the
  // longest tile under 3/4 of a share, where that is at least four; else four slots per SM (75 MB at D = 128) or that.
  const long long ntiles = (long long)B * Hkv * nKV;
  int heads = 1;
  while (heads < G && (G % heads != 0 || ntiles * heads < 2 * sms || longest * 4 * sms > 3 * total * heads)) ++heads;
  const long long room = heads > 1 ? ntiles * heads : 0;
  const long long budget = heads >= 4 ? room : std::max<long long>(room, 4ll * sms);
  while (pl.slots() > budget) --*std::max_element(pl.parts, pl.parts + 3);
  pl.choose_run(rest > 0 ? (double)(total - sinks) / rest * BQS / BQT : 0.0, reproducible);
  const double part = std::max((double)longest_sink / pl.run[0], (double)longest_rest / pl.run[1]);
  if (few && !reproducible && (part > 1.2 * share || (Nq <= 4096 && (long long)B * Hkv * G * Nq <= 81920))) pl.share_out(counts, nKV * Hkv, B, total, (int)longest);
  return pl;
}

// Packed batches: the lengths are on the device, so the plan goes by the average sequence.
BwdPlan bwd_plan_varlen(int B, int total, int Hkv, int G, const cowa_params_t* p, const CowaHeadWindows& hw) {
  BwdPlan pl;
  const int sms = cowa::sm_count(), len = std::max(total / B, 1);
  const long long rest = (long long)(total / BKV + B) * Hkv;
  pl.sink_tiles = 0;
  double keys = 0;
  for (int h = 0; h < Hkv; ++h) {
    CowaWin w = hw.w[h];
    if (p->full_attn) { w.s = 0; w.n = len; w.g = 0; w.l = 0; }
    else if (!p->windows) w = cowa_default_window(len, p->hkv_global > 0 ? p->hkv_global : Hkv, p->hkv_offset + h, p->sink, p->local);
    if (!p->full_attn) pl.sink_tiles = std::max(pl.sink_tiles, (std::min(p->windows ? w.s : p->sink, total) + BKV - 1) / BKV);
    keys += std::min<double>(len, (double)w.n + w.l + BKV) / Hkv;
  }
  pl.tiles[0] = B * Hkv * pl.sink_tiles;
  pl.parts[0] = pl.tiles[0] * 4ll <= 2 * sms ? 4 : 1;
  // the last wave is not shared here: short sequences make its tiles short already (1628 against 1624 in 1000 clocks)
  const double avg = 0.7 * keys / BQS * G, real = (double)total / BKV * Hkv;
  plan_rest(pl, rest, rest <= 2 * sms ? avg : 0.0, real * avg / sms);
  pl.choose_run(avg * BQS / BQT, p->deterministic != 0);
  return pl;
}

size_t slot_bytes(const BwdPlan& pl, int D) { return (size_t)pl.slots() * 2 * BKV * D * sizeof(float); }

size_t ws_bytes(int B, int Nq, int Hq, int D, const BwdPlan& pl) {
  const size_t Tpad = ((size_t)Nq + BQS - 1) / BQS * BQS;
  return (size_t)B * Hq * Tpad * ((size_t)D + 2) * sizeof(float) + slot_bytes(pl, D);
}

// Contiguous [H, T, D] (x batch) strides.
CowaStrides packed_strides(int H, long long T, int D) {
  CowaStrides st;
  st.t = D; st.h = T * D; st.b = (long long)H * T * D;
  return st;
}

// What comes behind the main kernel.
template <int D, bool VARLEN>
cudaError_t launch_finish(const BwdArgs& a, const BwdPlan& pl, const CowaStrides& sk, const CowaStrides& sv, void* dq_, int T,
                          const CowaStrides& sq, cudaStream_t st) {
  __nv_bfloat16* const dq = static_cast<__nv_bfloat16*>(dq_);
  const long long chunks = (long long)(a.Tpad / BQS) * a.Hq * (VARLEN ? 1 : a.B);
  long long shared = 0;
  for (int c = 0; c < 3; ++c)
    if (pl.run[c] > 1) shared += pl.tiles[c];
  if (pl.few > 0) shared = (long long)pl.few_shared * a.B;
  const long long sums = shared * kReduceBlocks<D>;
  if (sums > 0) {
    if (chunks <= kFinishChunks)
      return cowa::launch_chained(cowa_bwd_finish_kernel<D, VARLEN>, dim3((unsigned)(2 * sums + chunks)), 256, 0, st, a, sk, sv,
                                  (int)(2 * sums), dq, T, sq);
    cudaError_t e = cowa::launch_chained(cowa_bwd_reduce_dkv_kernel<D, VARLEN>, dim3((unsigned)sums, 2), 256, 0, st, a, sk, sv);
    if (e != cudaSuccess) return e;
  }
  return cowa::launch_chained(cowa_bwd_convert_dq_kernel<D, VARLEN>, dim3((unsigned)chunks), 256, 0, st, a.dq_acc, dq, a.cu, a.B, T,
                              a.Tpad, a.Hq, a.dq_fixed, sq, a.status);
}

template <int D>
int launch_bwd(const void* q, const void* k, const void* v, const void* o, const float* lse, const void* d_o,
               void* dq, void* dk, void* dv, int B, int Nq, int Nk, int Hq, int Hkv, const cowa_params_t* p,
               const CowaHeadWindows& hw, const BwdPlan& pl, void* ws, cudaStream_t st) {
  const int T = Nq;  // rows of q, o, d_o, dq, lse
  const int Tpad = (T + BQS - 1) / BQS * BQS;
  const long long BH = (long long)B * Hq;
  float* dq_acc = static_cast<float*>(ws);
  float* lse2 = dq_acc + (size_t)BH * Tpad * D;
  float* delta = lse2 + (size_t)BH * Tpad;
  float* dkv_part = delta + (size_t)BH * Tpad;
  // Everything that can fail is done before the first launch: strides, tensor maps, the status word.
  int rc;
  CowaStrides sq, sk, sv, so;
  if ((rc = cowa::resolve_strides(p->q_strides, Hq, Nq, D, &sq))) return rc;
  if ((rc = cowa::resolve_strides(p->k_strides, Hkv, Nk, D, &sk))) return rc;
  if ((rc = cowa::resolve_strides(p->v_strides, Hkv, Nk, D, &sv))) return rc;
  if ((rc = cowa::resolve_strides(p->o_strides, Hq, Nq, D, &so))) return rc;
  if (BH > 0x7FFFFFFFll) return COWA_ERR_UNSUPPORTED;
  CUtensorMap mq, mk, mv, mdo, mdk, mdv, mq2, mdo2;
  if ((rc = cowa::make_tensor_map(&mq, q, cowa::MapType::BF16, D, T, Hq, B, sq, 64, BQS))) return rc;
  if ((rc = cowa::make_tensor_map(&mq2, q, cowa::MapType::BF16, D, T, Hq, B, sq, 64, BQT))) return rc;
  if ((rc = cowa::make_tensor_map(&mdo, d_o, cowa::MapType::BF16, D, T, Hq, B, so, 64, BQS))) return rc;
  if ((rc = cowa::make_tensor_map(&mdo2, d_o, cowa::MapType::BF16, D, T, Hq, B, so, 64, BQT))) return rc;
  if ((rc = cowa::make_tensor_map(&mk, k, cowa::MapType::BF16, D, Nk, Hkv, B, sk, 64, BKV))) return rc;
  if ((rc = cowa::make_tensor_map(&mv, v, cowa::MapType::BF16, D, Nk, Hkv, B, sv, 64, BKV))) return rc;
  if ((rc = cowa::make_tensor_map(&mdk, dk, cowa::MapType::BF16, D, Nk, Hkv, B, sk, 64, BKV))) return rc;
  if ((rc = cowa::make_tensor_map(&mdv, dv, cowa::MapType::BF16, D, Nk, Hkv, B, sv, 64, BKV))) return rc;
  BwdArgs a;
  a.lse2 = lse2; a.delta = delta; a.dq_acc = dq_acc;
  a.status = cowa::device_status_word();
  if (!a.status) return COWA_ERR_CUDA;
  a.B = B; a.Nq = Nq; a.Nk = Nk; a.Hq = Hq; a.Hkv = Hkv; a.G = Hq / Hkv; a.Tpad = Tpad;
  a.scale = p->softmax_scale;
  a.scale_log2 = p->softmax_scale * 1.4426950408889634f;
  a.wins = hw;
  a.sink_tiles = pl.sink_tiles;
  for (int c = 0; c < 3; ++c) { a.cls_tiles[c] = pl.tiles[c]; a.cls_parts[c] = pl.run[c]; }
  a.single = pl.blocks() <= cowa::sm_count();
  a.few = pl.few;
  std::copy(pl.first, pl.first + pl.few + 1, a.first);
  std::copy(pl.shared, pl.shared + pl.few_shared, a.shared);
  a.dq_fixed = p->deterministic ? 1 : 0;
  a.dkv_part = dkv_part;
  a.cu = nullptr; a.dk = static_cast<__nv_bfloat16*>(dk); a.dv = static_cast<__nv_bfloat16*>(dv); a.total = 0; a.tiles_bound = 0;
  a.sdk = sk; a.sdv = sv;
  a.sink = 0; a.local = 0; a.hkv_global = 0; a.hkv_offset = 0; a.full_attn = 0; a.explicit_windows = 0;
  if (pl.blocks() > 0x7FFFFFFFll || (long long)Nq / BQS * a.G * 32 > 0x7FFFFFFFll) return COWA_ERR_UNSUPPORTED;
  COWA_CUDA_TRY(cudaFuncSetAttribute(cowa_bwd_kernel<D, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     BwdSmem<D>::kBytes));
  {
    const long long threads = BH * Tpad * (D / 8);
    COWA_CUDA_TRY(cowa::launch_chained(cowa_bwd_preprocess_kernel<D>, dim3((unsigned)((threads + 255) / 256)), 256, 0, st,
                                       static_cast<const __nv_bfloat16*>(o), static_cast<const __nv_bfloat16*>(d_o), lse,
                                       lse2, delta, dq_acc, T, Tpad, BH, Hq, so));
  }
  if (p->bwd_main_start_event) COWA_CUDA_TRY(cudaEventRecord(static_cast<cudaEvent_t>(p->bwd_main_start_event), st));
  COWA_CUDA_TRY(cowa::launch_chained(cowa_bwd_kernel<D, false>, dim3((unsigned)pl.blocks()), 512, BwdSmem<D>::kBytes, st, mq, mk, mv, mdo, mdk, mdv, mq2, mdo2, a));
  if (p->bwd_main_stop_event) COWA_CUDA_TRY(cudaEventRecord(static_cast<cudaEvent_t>(p->bwd_main_stop_event), st));
  COWA_CUDA_TRY((launch_finish<D, false>(a, pl, sk, sv, dq, T, sq, st)));
  return COWA_OK;
}

// Padded row space of a packed batch: every sequence rounded up to 64 rows; the bound needs no lengths.
int varlen_tpad(int B, int total) { return (total / BQS + B) * BQS; }

size_t ws_bytes_varlen(int B, int total, int Hq, int D, const BwdPlan& pl) {
  return (size_t)Hq * varlen_tpad(B, total) * ((size_t)D + 2) * sizeof(float) + slot_bytes(pl, D);
}

template <int D>
int launch_bwd_varlen(const void* q, const void* k, const void* v, const void* o, const float* lse, const void* d_o,
                      void* dq, void* dk, void* dv, const int* cu, int B, int total, int Hq, int Hkv,
                      const cowa_params_t* p, const CowaHeadWindows& hw, const BwdPlan& pl, void* ws, cudaStream_t st) {
  const int Tpad = varlen_tpad(B, total);
  float* dq_acc = static_cast<float*>(ws);
  float* lse2 = dq_acc + (size_t)Hq * Tpad * D;
  float* delta = lse2 + (size_t)Hq * Tpad;
  if (cowa::any_stride_set(p)) return COWA_ERR_UNSUPPORTED;  // packed tensors are contiguous [H, total, D]
  CUtensorMap mq, mk, mv, mdo, mdk, mdv, mq2, mdo2;
  int rc;
  const CowaStrides sq = packed_strides(Hq, total, D), sk = packed_strides(Hkv, total, D);
  if ((rc = cowa::make_tensor_map(&mq, q, cowa::MapType::BF16, D, total, Hq, 1, sq, 64, BQS))) return rc;
  if ((rc = cowa::make_tensor_map(&mq2, q, cowa::MapType::BF16, D, total, Hq, 1, sq, 64, BQT))) return rc;
  if ((rc = cowa::make_tensor_map(&mdo, d_o, cowa::MapType::BF16, D, total, Hq, 1, sq, 64, BQS))) return rc;
  if ((rc = cowa::make_tensor_map(&mdo2, d_o, cowa::MapType::BF16, D, total, Hq, 1, sq, 64, BQT))) return rc;
  if ((rc = cowa::make_tensor_map(&mk, k, cowa::MapType::BF16, D, total, Hkv, 1, sk, 64, BKV))) return rc;
  if ((rc = cowa::make_tensor_map(&mv, v, cowa::MapType::BF16, D, total, Hkv, 1, sk, 64, BKV))) return rc;
  if ((rc = cowa::make_tensor_map(&mdk, dk, cowa::MapType::BF16, D, total, Hkv, 1, sk, 64, BKV))) return rc;
  if ((rc = cowa::make_tensor_map(&mdv, dv, cowa::MapType::BF16, D, total, Hkv, 1, sk, 64, BKV))) return rc;
  BwdArgs a;
  a.lse2 = lse2; a.delta = delta; a.dq_acc = dq_acc;
  a.status = cowa::device_status_word();
  if (!a.status) return COWA_ERR_CUDA;
  a.B = B; a.Nq = 0; a.Nk = 0; a.Hq = Hq; a.Hkv = Hkv; a.G = Hq / Hkv; a.Tpad = Tpad;
  a.scale = p->softmax_scale;
  a.scale_log2 = p->softmax_scale * 1.4426950408889634f;
  a.wins = hw;
  a.sink_tiles = pl.sink_tiles;
  for (int c = 0; c < 3; ++c) { a.cls_tiles[c] = pl.tiles[c]; a.cls_parts[c] = pl.run[c]; }
  a.single = pl.blocks() <= cowa::sm_count();
  a.few = 0;
  a.dq_fixed = p->deterministic ? 1 : 0;
  a.dkv_part = delta + (size_t)Hq * Tpad;
  a.cu = cu; a.dk = static_cast<__nv_bfloat16*>(dk); a.dv = static_cast<__nv_bfloat16*>(dv);
  a.total = total; a.tiles_bound = total / BKV + B;
  a.sdk = a.sdv = sk;
  a.sink = p->sink; a.local = p->local;
  a.hkv_global = p->hkv_global > 0 ? p->hkv_global : Hkv;
  a.hkv_offset = p->hkv_offset; a.full_attn = p->full_attn; a.explicit_windows = p->windows != nullptr;
  if (pl.blocks() > 0x7FFFFFFFll || (long long)total / BQS * a.G * 32 > 0x7FFFFFFFll) return COWA_ERR_UNSUPPORTED;
  COWA_CUDA_TRY(cudaFuncSetAttribute(cowa_bwd_kernel<D, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     BwdSmem<D>::kBytes));
  const dim3 chunks(Tpad / BQS, Hq);
  COWA_CUDA_TRY(cowa::launch_chained(cowa_bwd_preprocess_varlen_kernel<D>, chunks, 256, 0, st,
                                     static_cast<const __nv_bfloat16*>(o), static_cast<const __nv_bfloat16*>(d_o), lse, lse2,
                                     delta, dq_acc, cu, B, total, Tpad, a.status));
  if (p->bwd_main_start_event) COWA_CUDA_TRY(cudaEventRecord(static_cast<cudaEvent_t>(p->bwd_main_start_event), st));
  COWA_CUDA_TRY(cowa::launch_chained(cowa_bwd_kernel<D, true>, dim3((unsigned)pl.blocks()), 512, BwdSmem<D>::kBytes, st, mq, mk, mv, mdo, mdk, mdv, mq2, mdo2, a));
  if (p->bwd_main_stop_event) COWA_CUDA_TRY(cudaEventRecord(static_cast<cudaEvent_t>(p->bwd_main_stop_event), st));
  COWA_CUDA_TRY((launch_finish<D, true>(a, pl, sk, sk, dq, total, sq, st)));
  return COWA_OK;
}

}  // namespace

extern "C" {

size_t cowa_bwd_varlen_workspace_bytes(int B, int total, int Hq, int Hkv, int D, const cowa_params_t* p) {
  if (B <= 0 || total <= 0 || Hq <= 0 || Hkv <= 0 || Hq % Hkv != 0 || (D != 64 && D != 128)) return 0;
  CowaHeadWindows hw;
  if (!p || cowa::resolve_windows(total, Hkv, p, &hw) != COWA_OK) {
    // Enough for any parameters: full attention has the most steps per tile, hence parts; and as many sink tiles as are
    // shared at all (bwd_plan_varlen).
    cowa_params_t full = {};
    full.full_attn = 1;
    BwdPlan most = bwd_plan_varlen(B, total, Hkv, Hq / Hkv, &full, hw);
    most.tiles[0] = std::min(cowa::sm_count() / 2, (int)std::min<long long>((long long)B * Hkv * ((total + BKV - 1) / BKV), 1 << 20));
    most.parts[0] = 4;
    return ws_bytes_varlen(B, total, Hq, D, most);
  }
  return ws_bytes_varlen(B, total, Hq, D, bwd_plan_varlen(B, total, Hkv, Hq / Hkv, p, hw));
}

int cowa_bwd_varlen(const void* q, const void* k, const void* v, const void* o, const float* lse, const void* d_o,
                    void* dq, void* dk, void* dv, const int32_t* cu_seqlens, int B, int total, int Hq, int Hkv, int D,
                    const cowa_params_t* p, void* workspace, size_t workspace_bytes, void* stream) {
  if (!q || !k || !v || !o || !lse || !d_o || !dq || !dk || !dv || !p || !workspace || !cu_seqlens)
    return COWA_ERR_INVALID_ARG;
  if (B <= 0 || total <= 0 || Hq <= 0 || Hkv <= 0 || Hq % Hkv != 0) return COWA_ERR_INVALID_ARG;
  if (!(p->softmax_scale > 0.f)) return COWA_ERR_INVALID_ARG;
  if (D != 64 && D != 128) return COWA_ERR_UNSUPPORTED;
  const void* ptrs[] = {q, k, v, o, d_o, dq, dk, dv, workspace};
  for (const void* x : ptrs)
    if (!cowa::aligned16(x)) return COWA_ERR_MISALIGNED;
  CowaHeadWindows hw;
  int rc = cowa::resolve_windows(total, Hkv, p, &hw);  // validates; explicit tuples are copied, the default rule runs per sequence
  if (rc != COWA_OK) return rc;
  const BwdPlan pl = bwd_plan_varlen(B, total, Hkv, Hq / Hkv, p, hw);
  if (workspace_bytes < ws_bytes_varlen(B, total, Hq, D, pl)) return COWA_ERR_WORKSPACE_TOO_SMALL;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  return D == 128 ? launch_bwd_varlen<128>(q, k, v, o, lse, d_o, dq, dk, dv, cu_seqlens, B, total, Hq, Hkv, p, hw,
                                           pl, workspace, st)
                  : launch_bwd_varlen<64>(q, k, v, o, lse, d_o, dq, dk, dv, cu_seqlens, B, total, Hq, Hkv, p, hw,
                                          pl, workspace, st);
}

size_t cowa_bwd_prefill_workspace_bytes(int B, int Nq, int Nk, int Hq, int Hkv, int D, const cowa_params_t* p) {
  if (B <= 0 || Nq <= 0 || Nk < Nq || Hq <= 0 || Hkv <= 0 || Hq % Hkv != 0 || D <= 0 || !p) return 0;
  CowaHeadWindows hw;
  if (cowa::resolve_windows(Nk, Hkv, p, &hw) != COWA_OK) return 0;
  return ws_bytes(B, Nq, Hq, D, bwd_plan(B, Nq, Nk, Hkv, Hq / Hkv, hw, p->deterministic != 0));
}

size_t cowa_bwd_workspace_bytes(int B, int T, int Hq, int Hkv, int D, const cowa_params_t* p) {
  return cowa_bwd_prefill_workspace_bytes(B, T, T, Hq, Hkv, D, p);
}

int cowa_bwd_prefill(const void* q, const void* k, const void* v, const void* o, const float* lse, const void* d_o,
                     void* dq, void* dk, void* dv, int B, int Nq, int Nk, int Hq, int Hkv, int D,
                     const cowa_params_t* p, void* workspace, size_t workspace_bytes, void* stream) {
  if (!q || !k || !v || !o || !lse || !d_o || !dq || !dk || !dv || !p || !workspace) return COWA_ERR_INVALID_ARG;
  if (B <= 0 || Nq <= 0 || Nk < Nq || Hq <= 0 || Hkv <= 0 || Hq % Hkv != 0) return COWA_ERR_INVALID_ARG;
  if (!(p->softmax_scale > 0.f)) return COWA_ERR_INVALID_ARG;
  if (D != 64 && D != 128) return COWA_ERR_UNSUPPORTED;
  const void* ptrs[] = {q, k, v, o, d_o, dq, dk, dv, workspace};
  for (const void* x : ptrs)
    if (!cowa::aligned16(x)) return COWA_ERR_MISALIGNED;
  CowaHeadWindows hw;
  int rc = cowa::resolve_windows(Nk, Hkv, p, &hw);
  if (rc != COWA_OK) return rc;
  const BwdPlan pl = bwd_plan(B, Nq, Nk, Hkv, Hq / Hkv, hw, p->deterministic != 0);
  if (workspace_bytes < ws_bytes(B, Nq, Hq, D, pl)) return COWA_ERR_WORKSPACE_TOO_SMALL;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  return D == 128 ? launch_bwd<128>(q, k, v, o, lse, d_o, dq, dk, dv, B, Nq, Nk, Hq, Hkv, p, hw, pl, workspace, st)
                  : launch_bwd<64>(q, k, v, o, lse, d_o, dq, dk, dv, B, Nq, Nk, Hq, Hkv, p, hw, pl, workspace, st);
}

int cowa_bwd(const void* q, const void* k, const void* v, const void* o, const float* lse, const void* d_o,
             void* dq, void* dk, void* dv, int B, int T, int Hq, int Hkv, int D, const cowa_params_t* p,
             void* workspace, size_t workspace_bytes, void* stream) {
  return cowa_bwd_prefill(q, k, v, o, lse, d_o, dq, dk, dv, B, T, T, Hq, Hkv, D, p, workspace, workspace_bytes, stream);
}

}  // extern "C"
