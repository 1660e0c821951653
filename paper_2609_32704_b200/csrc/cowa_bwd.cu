// CoWindow Attention backward (Algorithm 2) for sm_100a.
//
// Three launches on the caller's stream, four when some KV tiles are shared:
//   1. preprocess   -Delta = -rowsum(O * dO) (Algorithm 2 line 13) and -LSE * log2(e), fp32 row vectors
//                   padded to a multiple of 64 rows (padding: -inf, so that P = 0 there);
//                   its threads also zero the fp32 dQ accumulator.
//   2. main kernel  one thread block per (batch, KV head, 128-row KV tile), KV-stationary as in
//                   Algorithm 2, looping over the G QO heads of the group and over the 64-row QO
//                   tiles of I_h(j) (analytic scheduler, ascending).  Per step five tcgen05 MMAs:
//                     S^T  = K Q^T            (TMEM, 128 kv x 64 q)
//                     dP^T = V dO^T           (TMEM)
//                     dV  += P^T dO           (P^T as the TMEM operand)
//                     dK  += dS^T Q           (dS^T as the TMEM operand)
//                     dQ^T = K^T dS^T         (dS^T from shared memory; 128 d x 64 q in TMEM)
//                   dK and dV stay in TMEM for the whole loop, all G heads included, so they need no
//                   atomics (Algorithm 2 line 17 needs them only because it gives each QO head its
//                   own program).  dQ^T is drained by a separate warpgroup through shared memory and
//                   added to the fp32 accumulator with bulk add-reductions of contiguous 32-row ranges (Algorithm 2 line 15).
//                   Warp roles: TMA producer / MMA issuer / two compute warpgroups (P, dS; each takes 32
//                   of the 64 query columns of every step, which halves the latency between S^T and
//                   dS^T) / dQ drain warpgroup, connected by mbarriers; S^T is double buffered so that the
//                   MMAs of steps n+1, n+2 overlap the element-wise work of
//                   step n.  Blocks are ordered sink tiles first (they meet every query tile), then
//                   head by head with ascending KV tile, so that the blocks in flight sweep the same
//                   dQ rows at nearly the same time and the reductions hit in L2.
//   3. convert      dQ accumulator (already scaled) -> bf16.
// Two variations of the main kernel's work split:
//   - shared tiles: a tile's steps are cut into contiguous parts for several blocks (few tiles, sink tiles that would
//     be the critical path, the last wave); each block writes fp32 partial dK, dV to its own slot and a
//     fourth kernel adds the slots in order (BwdPlan).
//   - VARLEN: packed batch [H, total, D]; a block finds (sequence, KV tile) by a warp scan of the offsets,
//     windows follow from the sequence's own length, the accumulator and the row vectors use a row space
//     in which every sequence is padded to 64 rows, and a sequence's last, partial KV tile is stored row
//     by row (cowa_bwd_varlen and its own preprocess / convert kernels).
#include <cuda_bf16.h>

#include <algorithm>
#include <type_traits>

#include "cowa_common.h"
#include "cowa_ptx.cuh"
#include "cowa_tma.h"

using namespace cowa_ptx;

namespace {

constexpr int BKV = 128;  // KV rows per block (MMA M)
constexpr int BQS = 64;   // QO rows per step (MMA N of S^T / dP^T)
constexpr int NST = 3;    // Q / dO stages
constexpr float kDqFixedOne = 262144.f;  // 2^18: one unit of dQ in the fixed-point accumulation mode

struct BwdArgs {
  const float* lse2;   // [B*Hq, Tpad]  -LSE * log2(e)   (both negated: the packed adds have no operand negation)
  const float* delta;  // [B*Hq, Tpad]  -Delta
  float* dq_acc;       // [B*Hq, Tpad, D] fp32
  unsigned int* status;
  int B, Nq, Nk, Hq, Hkv, G, Tpad;
  int sink_tiles;      // KV tiles per head that hold sink columns (launched first)
  // The KV tiles in launch order: sink tiles, body, tail.  A tile of class c is shared by cls_parts[c] blocks, each with
  // a contiguous part of the tile's steps (QO heads x QO tiles); a shared tile's blocks leave fp32 partial dK, dV.
  int cls_tiles[3], cls_parts[3];
  int dq_fixed;        // 1: dQ partial sums travel as 32-bit fixed point (order-independent addition)
  float* dkv_part;     // fp32 partial dK, dV [blocks of shared tiles, 2, BKV, D], summed by a kernel of their own
  // packed (variable-length) batches only: tensors are [H, total, D], sequence b owns rows cu[b] .. cu[b+1]
  const int* cu;       // [B+1] device
  __nv_bfloat16* dk;   // raw outputs for the last, partial KV tile of a sequence
  __nv_bfloat16* dv;
  int total, tiles_bound;  // rows of the packed tensors; grid tiles per KV head (upper bound of the real count)
  int sink, local, hkv_global, hkv_offset, full_attn, explicit_windows;
  float scale, scale_log2;
  CowaHeadWindows wins;
};

template <int D>
struct BwdSmem {
  static constexpr int kKV = BKV * D * 2;      // K or V tile
  static constexpr int kQS = BQS * D * 2;      // Q or dO step tile
  static constexpr int kStage = 2 * kQS;       // Q + dO
  static constexpr int kDS = BKV * BQS * 2;    // dS^T tile (bf16)
  static constexpr int oK = 0, oV = kKV, oStage = 2 * kKV, oDS = oStage + NST * kStage;
  static constexpr int oVec = oDS + 2 * kDS;   // per stage: 64 floats lse2, 64 floats delta
  static constexpr int oDQ = oVec + NST * 512;  // dQ staging: two tiles of 32 query rows x D fp32
  static constexpr int kDQ = 32 * D * 4;
  static constexpr int oBar = oDQ + 2 * kDQ;
  static constexpr int kBytes = oBar + 256 + 1024;  // barriers + alignment slack; 232192 B at D = 128 (limit 232448)
};

__device__ __forceinline__ void bulk_load_1d(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_u32(dst)),
               "l"(src), "r"(bytes), "r"(smem_u32(bar))
               : "memory");
}

__device__ __forceinline__ void bulk_store(void* dst, const void* src, uint32_t bytes) {
  asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst), "r"(smem_u32(src)), "r"(bytes)
               : "memory");
}

__device__ __forceinline__ uint32_t interval_bits32(long long a, long long b, long long base) {
  long long lo = a - base, hi = b - base;
  if (lo < 0) lo = 0;
  if (hi > 31) hi = 31;
  if (lo > hi) return 0u;
  return (0xFFFFFFFFu >> (31 - (int)(hi - lo))) << (int)lo;
}

// Tile number q of class c: sink tiles of every head first (they meet every query tile of their sequence and are the
// longest), then head-major with ascending KV tile (consecutive blocks share dQ rows, which then stay in L2).  Packed
// batches: whole warps only; false when there is no such tile (the count is an upper bound).
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
    x.hk = q / a.tiles_bound;
    return varlen_locate(a.cu, a.B, q % a.tiles_bound, BKV, BQS, &x.b, &x.j, &x.nts, &x.pbase, nsk) && fits(a, x);
  }
  const int nrest = (a.Nk + BKV - 1) / BKV - nsk;
  x.j = nsk + q % nrest; q /= nrest;
  x.hk = q % a.Hkv; x.b = q / a.Hkv;
  return true;
}

// named barrier for one 128-thread warpgroup
__device__ __forceinline__ void wg_sync(int id) { asm volatile("bar.sync %0, 128;" ::"r"(id) : "memory"); }

template <int D, bool VARLEN>
__global__ void __launch_bounds__(512, 1)
cowa_bwd_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                const __grid_constant__ CUtensorMap tmV, const __grid_constant__ CUtensorMap tmdO,
                const __grid_constant__ CUtensorMap tmdK, const __grid_constant__ CUtensorMap tmdV,
                const __grid_constant__ BwdArgs a) {
  using SM = BwdSmem<D>;
  constexpr int NSLAB = D / 64;
  constexpr int SLAB_KV = BKV * 128;  // bytes of one 64-wide slab of a 128-row tile
  constexpr int SLAB_QS = BQS * 128;  // ... of a 64-row tile
  // TMEM columns
  constexpr uint32_t cS0 = 0, cDP0 = 128, cDK = 256, cDV = 384, TMEM_COLS = 512;  // S^T x2, dP^T/dQ^T x2, dK, dV
  constexpr uint32_t ID_ST = idesc_bf16(128, BQS, 0, 0);   // S^T, dP^T
  constexpr uint32_t ID_ACC = idesc_bf16(128, D, 0, 1);    // dV, dK (B = dO / Q, MN-major)
  constexpr uint32_t ID_DQ = idesc_bf16(128, BQS, 1, 1);   // dQ^T (A = K^T, B = dS^T, both MN-major)

  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* sK = smem + SM::oK;
  uint8_t* sV = smem + SM::oV;
  uint8_t* sStage = smem + SM::oStage;
  uint8_t* sDS = smem + SM::oDS;
  float* sVec = reinterpret_cast<float*>(smem + SM::oVec);
  float* sDQ = reinterpret_cast<float*>(smem + SM::oDQ);
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + SM::oBar);
  uint64_t* bar_kv = bars + 0;
  uint64_t* bar_ld_full = bars + 1;             // [NST]  Q/dO/LSE/Delta of a step have landed
  uint64_t* bar_ld_empty = bars + 1 + NST;      // [NST]  the step's products have consumed the stage
  uint64_t* bar_s_full = bars + 1 + 2 * NST;    // [2]    S^T of a step is in TMEM buffer b
  uint64_t* bar_dp_full = bars + 3 + 2 * NST;   // [2]    dP^T ...
  uint64_t* bar_p_ready = bars + 5 + 2 * NST;   // [2]    count 256: P^T written over S^T
  uint64_t* bar_ds_ready = bars + 7 + 2 * NST;  // [2]    count 256: dS^T in TMEM and shared memory, dP^T consumed
  uint64_t* bar_dq_full = bars + 9 + 2 * NST;   // [2]    dQ^T is in the columns dP^T left
  uint64_t* bar_dq_free = bars + 11 + 2 * NST;  // [2]    count 128: dQ^T drained
  uint64_t* bar_done = bars + 13 + 2 * NST;
  uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(bars + 14 + 2 * NST);
  float** part_out = reinterpret_cast<float**>(bars + 15 + 2 * NST);  // this block's partial dK, dV (kept here, not in registers)

  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);  // warp-uniform by construction (helps the compiler)

  // ---- work item ----
  int cls = 0, idx = blockIdx.x, slot = 0;
  while (cls < 2 && idx >= a.cls_tiles[cls] * a.cls_parts[cls]) {
    idx -= a.cls_tiles[cls] * a.cls_parts[cls];
    if (a.cls_parts[cls] > 1) slot += a.cls_tiles[cls] * a.cls_parts[cls];
    ++cls;
  }
  const int parts = a.cls_parts[cls], part = idx % parts;
  slot += idx;  // of this block's partial dK, dV when the tile is shared
  TileAt at;
  if (!locate_tile<VARLEN>(a, cls, idx / parts, at)) return;
  const int hk = at.hk, b = at.b, j = at.j, pbase = at.pbase;
  // Sequence geometry.  Packed batches: N_q = N_k = the sequence's length, rows start at cu[b]; the fp32
  // dQ accumulator and the LSE / Delta vectors are laid out with every sequence padded to 64 rows (pbase).
  int Nq = a.Nq, Nk = a.Nk, rbase = 0;
  CowaWin w = a.wins.w[hk];
  if constexpr (VARLEN) {
    rbase = a.cu[b];
    Nq = Nk = a.cu[b + 1] - rbase;
    if (rbase < 0 || rbase + Nk > a.total) {  // malformed offsets: report, touch nothing
      if (threadIdx.x == 0) atomicOr(a.status, (unsigned)COWA_DEV_BAD_SEQLENS);
      return;
    }
    if (a.full_attn) { w.s = 0; w.n = Nk; w.g = 0; w.l = 0; }
    else if (!a.explicit_windows) w = cowa_default_window(Nk, a.hkv_global, a.hkv_offset + hk, a.sink, a.local);
  }
  const int off = Nk - Nq;
  const int k0 = j * BKV, k1 = min(k0 + BKV, Nk) - 1;
  CowaRange rg[2];
  cowa_bwd_ranges(w, k0, k1, off, Nq, BQS, rg);
  const int cnt = cowa_range_len(rg[0]) + cowa_range_len(rg[1]);  // QO steps per head
  const int n0 = cnt * a.G * part / parts;               // (the host checks that these products fit)
  const int N = cnt * a.G * (part + 1) / parts - n0;     // this block's steps
  const int g0 = cnt > 0 ? n0 / cnt : 0, tq0 = n0 - g0 * cnt;  // head of the group and position in I_h(j) of the first
  const int bt = VARLEN ? 0 : b;                               // batch coordinate of the tensor maps
  const int hq0 = hk * a.G;                                    // first QO head of the group
  const int bhq0 = (VARLEN ? 0 : b * a.Hq) + hq0;              // ... as a row of lse2 / delta / dq_acc
  const size_t vec_stride = (size_t)a.Tpad;                                         // rows per head in lse2 / delta / dq_acc
  const bool tail_kv = VARLEN && (k0 + BKV > Nk);  // rows after the tile's last valid one belong to the next sequence

  if (tid == 0) {
    *part_out = parts > 1 ? a.dkv_part + (size_t)slot * 2 * (BKV * D) : nullptr;
    mbar_init(bar_kv, 1);
    for (int s = 0; s < NST; ++s) { mbar_init(bar_ld_full + s, 1); mbar_init(bar_ld_empty + s, 1); }
    for (int s = 0; s < 2; ++s) {
      mbar_init(bar_s_full + s, 1); mbar_init(bar_dp_full + s, 1);
      mbar_init(bar_p_ready + s, 256); mbar_init(bar_ds_ready + s, 256);
      mbar_init(bar_dq_full + s, 1); mbar_init(bar_dq_free + s, 128);
    }
    mbar_init(bar_done, 1);
    fence_mbar_init();
  }
  if (warp == 0) {
    __syncwarp();
    tmem_alloc(tmem_holder, TMEM_COLS);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_holder;

  bool ok = true;

  // dK (first compute warpgroup) and dV (drain warpgroup): TMEM -> bf16 -> shared -> TMA store.  Called from
  // inside the role branches so that it is compiled under that role's register budget.
  auto store_grad = [&](bool is_dk) {
    const int r = (warp & 3) * 32 + lane;
    const uint32_t t_lane = tmem_base + ((uint32_t)((warp & 3) * 32) << 16);
    if (N > 0) ok = mbar_wait(bar_done, 0, a.status) && ok;
    tc_fence_after();
    uint8_t* sOut = sStage + (is_dk ? 0 : SM::kKV);
    const float mul = is_dk ? a.scale : 1.f;
    if (float* const dst = *part_out) {
      // A shared tile: this block's part goes out in fp32, one slot per block; a kernel of its own adds the slots in order.
      // Staged where K, V or the Q / dO stages were, rows with their 16-byte chunks permuted (bank conflicts), and
      // copied as one range: straight from registers a warp's store touches 32 rows (1019 against 983 thousand clocks of
      // the whole kernel for one KV head of 20001 tokens).
      uint8_t* sPart = (is_dk ? sK : sStage) + r * (D * 4);
#pragma unroll
      for (int c = 0; c < D / 32; ++c) {
        uint32_t ov[32];
        if (N > 0 && ok) {
          tmem_ld32(t_lane + (is_dk ? cDK : cDV) + c * 32, ov);
          tmem_wait_ld();
        } else {
#pragma unroll
          for (int e = 0; e < 32; ++e) ov[e] = 0u;
        }
#pragma unroll
        for (int q = 0; q < 8; ++q)
          *reinterpret_cast<float4*>(sPart + (((c * 8 + q) ^ (r & 7)) << 4)) =
              make_float4(__uint_as_float(ov[q * 4]) * mul, __uint_as_float(ov[q * 4 + 1]) * mul,
                          __uint_as_float(ov[q * 4 + 2]) * mul, __uint_as_float(ov[q * 4 + 3]) * mul);
      }
      fence_proxy_async_smem();
      wg_sync(is_dk ? 1 : 2);
      if (r == 0) {
        bulk_store(dst + (is_dk ? 0 : BKV * D), is_dk ? sK : sStage, BKV * D * 4);
        tma_commit_group();
        tma_wait_group<0>();
      }
      return;
    }
    if (tail_kv) {
      // last, partial KV tile of a packed sequence: row by row, straight from registers
      __nv_bfloat16* dst = (is_dk ? a.dk : a.dv) + ((size_t)hk * a.total + rbase + k0 + r) * D;
#pragma unroll
      for (int c = 0; c < D / 32; ++c) {
        uint32_t ov[32];
        if (N > 0 && ok) {
          tmem_ld32(t_lane + (is_dk ? cDK : cDV) + c * 32, ov);
          tmem_wait_ld();
        } else {
#pragma unroll
          for (int e = 0; e < 32; ++e) ov[e] = 0u;
        }
        if (k0 + r < Nk) {
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            uint4 v;
            v.x = pack_bf16(__uint_as_float(ov[q * 8 + 0]) * mul, __uint_as_float(ov[q * 8 + 1]) * mul);
            v.y = pack_bf16(__uint_as_float(ov[q * 8 + 2]) * mul, __uint_as_float(ov[q * 8 + 3]) * mul);
            v.z = pack_bf16(__uint_as_float(ov[q * 8 + 4]) * mul, __uint_as_float(ov[q * 8 + 5]) * mul);
            v.w = pack_bf16(__uint_as_float(ov[q * 8 + 6]) * mul, __uint_as_float(ov[q * 8 + 7]) * mul);
            *reinterpret_cast<uint4*>(dst + c * 32 + q * 8) = v;
          }
        }
      }
      return;
    }
#pragma unroll
    for (int c = 0; c < D / 32; ++c) {
      uint32_t ov[32];
      if (N > 0 && ok) {
        tmem_ld32(t_lane + (is_dk ? cDK : cDV) + c * 32, ov);
        tmem_wait_ld();
      } else {
#pragma unroll
        for (int e = 0; e < 32; ++e) ov[e] = 0u;
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        uint4 v;
        v.x = pack_bf16(__uint_as_float(ov[q * 8 + 0]) * mul, __uint_as_float(ov[q * 8 + 1]) * mul);
        v.y = pack_bf16(__uint_as_float(ov[q * 8 + 2]) * mul, __uint_as_float(ov[q * 8 + 3]) * mul);
        v.z = pack_bf16(__uint_as_float(ov[q * 8 + 4]) * mul, __uint_as_float(ov[q * 8 + 5]) * mul);
        v.w = pack_bf16(__uint_as_float(ov[q * 8 + 6]) * mul, __uint_as_float(ov[q * 8 + 7]) * mul);
        const int d0 = c * 32 + q * 8;
        const int slab = d0 / 64, chunk = (d0 % 64) / 8;
        *reinterpret_cast<uint4*>(sOut + slab * SLAB_KV + r * 128 + ((chunk ^ (r & 7)) << 4)) = v;
      }
    }
    fence_proxy_async_smem();
    wg_sync(is_dk ? 1 : 2);
    if (r == 0 && ok) {
      for (int s = 0; s < NSLAB; ++s) tma_store_4d(is_dk ? &tmdK : &tmdV, sOut + s * SLAB_KV, s * 64, rbase + k0, hk, bt);
      tma_commit_group();
      tma_wait_group<0>();
    }
  };

  // Register budget per role: 128 per thread at launch (512 threads), 80 + 2 * 160 + 112 = 4 * 128 moved to where the work
  // is.  Each setmaxnreg sits at the top of its own branch so that the code below it is compiled for that budget.  No
  // role spills at these: with 64 / 176 / 96 the MMA issuer and the producer did, inside their loops, and the kernel took
  // 1066 instead of 1015 thousand clocks at 2 x 8K, 7980 instead of 7590 at 32K.
  if (warp < 4) {
    setmaxnreg_dec<80>();
    if (warp == 0) {
      // ================= TMA producer =================
      if (lane == 0 && N > 0) {
        prefetch_tmap(&tmQ); prefetch_tmap(&tmdO); prefetch_tmap(&tmK); prefetch_tmap(&tmV);
        mbar_expect_tx(bar_kv, 2 * SM::kKV);
        for (int s = 0; s < NSLAB; ++s) {
          tma_load_4d(sK + s * SLAB_KV, &tmK, bar_kv, s * 64, rbase + k0, hk, bt);
          tma_load_4d(sV + s * SLAB_KV, &tmV, bar_kv, s * 64, rbase + k0, hk, bt);
        }
        int st = 0, g = g0, t_in = tq0;   // stage, head of the group, position in I_h(j): kept incrementally
        uint32_t ph_e = 0;             // parity of the "stage empty" wait (the first NST steps need none)
        for (int n = 0; n < N && ok; ++n) {
          if (n >= NST) ok = mbar_wait(bar_ld_empty + st, ph_e, a.status);
          if (!ok) break;
          const int i = cowa_bwd_tile_at(rg, t_in);
          const int bhq = bhq0 + g, q0 = i * BQS;
          uint8_t* sQ = sStage + st * SM::kStage;
          uint8_t* sdO = sQ + SM::kQS;
          mbar_expect_tx(bar_ld_full + st, SM::kStage + 512);
          for (int s = 0; s < NSLAB; ++s) {
            tma_load_4d(sQ + s * SLAB_QS, &tmQ, bar_ld_full + st, s * 64, rbase + q0, hq0 + g, bt);
            tma_load_4d(sdO + s * SLAB_QS, &tmdO, bar_ld_full + st, s * 64, rbase + q0, hq0 + g, bt);
          }
          bulk_load_1d(sVec + st * 128, a.lse2 + (size_t)bhq * vec_stride + pbase + q0, 256, bar_ld_full + st);
          bulk_load_1d(sVec + st * 128 + 64, a.delta + (size_t)bhq * vec_stride + pbase + q0, 256, bar_ld_full + st);
          if (++t_in == cnt) { t_in = 0; ++g; }
          if (++st == NST) { st = 0; if (n >= NST) ph_e ^= 1; }
        }
      }
    } else if (warp == 1) {
      // ================= MMA issuer =================
      // The whole warp runs this loop (uniform control flow, so that descriptors and counters stay in
      // uniform registers); only the elected lane executes the tcgen05 instructions.  Everything that
      // can be computed once is: descriptor of every operand base, stage and parity bookkeeping is
      // incremental, and the loop body is instantiated for both TMEM buffers.
      if (N > 0) {
        const bool lead = elect_one();
        const uint32_t tb = tmem_base;
        // Descriptors: a byte offset o inside a tile is added as o >> 4 to the address field (bits 0-13);
        // no tile crosses the field's range, so the 64-bit add never carries out of it.
        const uint64_t dK_k = smem_desc_sw128(smem_u32(sK), 16, 1024);                       // K, K-major (A of S^T)
        const uint64_t dV_k = smem_desc_sw128(smem_u32(sV), 16, 1024);                       // V, K-major (A of dP^T)
        const uint64_t dK_mn = smem_desc_sw128(smem_u32(sK), D == 128 ? SLAB_KV : 0, 1024);  // K^T, MN-major (A of dQ^T)
        const uint64_t dQ_k0 = smem_desc_sw128(smem_u32(sStage), 16, 1024);                  // Q of stage 0, K-major (B of S^T)
        const uint64_t dO_k0 = smem_desc_sw128(smem_u32(sStage) + SM::kQS, 16, 1024);        // dO of stage 0, K-major (B of dP^T)
        const uint64_t dQ_mn0 = smem_desc_sw128(smem_u32(sStage), SLAB_QS, 1024);            // Q, MN-major (B of dK)
        const uint64_t dO_mn0 = smem_desc_sw128(smem_u32(sStage) + SM::kQS, SLAB_QS, 1024);  // dO, MN-major (B of dV)
        const uint64_t dDS0 = smem_desc_sw128(smem_u32(sDS), 0, 1024);                       // dS^T, MN-major (B of dQ^T)
        constexpr uint32_t kStage16 = SM::kStage >> 4, kDS16 = SM::kDS >> 4;

        auto gemm_st = [&](uint32_t d_col, uint64_t dA, uint64_t dB) {  // [128 x 64] = A[128 x D] B[64 x D]^T
          if (lead) {
#pragma unroll
            for (int kk = 0; kk < D / 16; ++kk)
              mma_ss(tb + d_col, dA + (((kk / 4) * SLAB_KV + (kk % 4) * 32) >> 4),
                     dB + (((kk / 4) * SLAB_QS + (kk % 4) * 32) >> 4), ID_ST, kk > 0);
          }
        };
        auto gemm_acc = [&](uint32_t d_col, uint32_t a_col, uint64_t dB, uint32_t acc_first) {  // [128 x D] += A(TMEM) B
          if (lead) {
#pragma unroll
            for (int kk = 0; kk < BQS / 16; ++kk)
              mma_ts(tb + d_col, tb + a_col + (kk >> 1) * 32 + (kk & 1) * 8, dB + ((kk * 2048) >> 4), ID_ACC, kk > 0 ? 1u : acc_first);
          }
        };
        auto gemm_dq = [&](uint32_t d_col, uint64_t dB) {  // dQ^T[D x 64] = K^T dS^T
          if (lead) {
#pragma unroll
            for (int kk = 0; kk < BKV / 16; ++kk)
              mma_ss(tb + d_col, dK_mn + ((kk * 2048) >> 4), dB + ((kk * 2048) >> 4), ID_DQ, kk > 0);
          }
        };
        auto commit = [&](uint64_t* bar) {
          if (lead) mma_commit(bar);
        };

        // Packed batches: rows of a tile that lie past the end of the sequence belong to the next one.  Every
        // product they enter is multiplied by an exact zero, but 0 x (Inf or NaN) would still poison this
        // sequence, so they are cleared in shared memory (whole 128-byte rows, by this warp) before use.
        auto clear_rows = [&](uint8_t* tile, int first, int rows, int slab_bytes) {
          const int nchunk = (rows - first) * 8;  // 16-byte chunks per slab
          for (int s_ = 0; s_ < NSLAB; ++s_)
            for (int c_ = lane; c_ < nchunk; c_ += 32)
              *reinterpret_cast<uint4*>(tile + s_ * slab_bytes + first * 128 + c_ * 16) = make_uint4(0u, 0u, 0u, 0u);
        };
        int t_clr = tq0;  // position in I_h(j) of the next step whose Q / dO stage is checked (packed batches only)
        auto clear_stage_tail = [&](int stage) {
          if constexpr (VARLEN) {
            const int q0_ = cowa_bwd_tile_at(rg, t_clr) * BQS;
            if (++t_clr == cnt) t_clr = 0;
            if (q0_ + BQS > Nq) {
              uint8_t* sQ_ = sStage + stage * SM::kStage;
              clear_rows(sQ_, Nq - q0_, BQS, SLAB_QS);
              clear_rows(sQ_ + SM::kQS, Nq - q0_, BQS, SLAB_QS);
              fence_proxy_async_smem();
              __syncwarp();
            }
          }
        };
        ok = mbar_wait(bar_kv, 0, a.status);
        if (ok && tail_kv) {
          clear_rows(sK, Nk - k0, BKV, SLAB_KV);
          clear_rows(sV, Nk - k0, BKV, SLAB_KV);
          fence_proxy_async_smem();
          __syncwarp();
        }
        // prologue: S^T(0), dP^T(0), S^T(1)
        ok = ok && mbar_wait(bar_ld_full + 0, 0, a.status);
        if (ok) {
          clear_stage_tail(0);
          tc_fence_after();
          gemm_st(cS0, dK_k, dQ_k0);
          commit(bar_s_full + 0);
          gemm_st(cDP0, dV_k, dO_k0);
          commit(bar_dp_full + 0);
        }
        if (ok && N > 1) {
          ok = mbar_wait(bar_ld_full + 1, 0, a.status);
          if (ok) {
            clear_stage_tail(1);
            tc_fence_after();
            gemm_st(cS0 + 64, dK_k, dQ_k0 + kStage16);
            commit(bar_s_full + 1);
          }
        }
        // Step n uses TMEM buffer b = n & 1.  Issue order:
        //   dV(n) | dP^T(n+1) | dK(n) | S^T(n+2) | dQ^T(n)
        // so that every wait below is for something produced about one step earlier.
        int st = 0, st1 = (N > 1) ? 1 : 0, st2 = 2 % NST;    // stages of steps n, n+1, n+2
        uint32_t ph2 = (2 / NST) & 1;                        // parity of the load that fills stage st2 for step n+2
        uint32_t par = 0;                                    // (n >> 1) & 1
        auto body = [&](int n, auto B_) {
          constexpr int b_ = decltype(B_)::value;
          constexpr uint32_t sbuf = cS0 + b_ * 64, dpbuf = cDP0 + b_ * 64, dpother = cDP0 + (b_ ^ 1) * 64;
          ok = mbar_wait(bar_p_ready + b_, par, a.status);
          if (!ok) return;
          tc_fence_after();
          gemm_acc(cDV, sbuf, dO_mn0 + st * kStage16, n > 0 ? 1u : 0u);     // dV += P^T dO
          if (n + 1 < N) {                                                  // dP^T(n+1), once dQ^T(n-1) has left its buffer
            if (n >= 1) {
              ok = mbar_wait(bar_dq_free + (b_ ^ 1), ((n - 1) >> 1) & 1, a.status);
              if (!ok) return;
              tc_fence_after();
            }
            gemm_st(dpother, dV_k, dO_k0 + st1 * kStage16);
            commit(bar_dp_full + (b_ ^ 1));
          }
          ok = mbar_wait(bar_ds_ready + b_, par, a.status);
          if (!ok) return;
          tc_fence_after();
          gemm_acc(cDK, sbuf + 16, dQ_mn0 + st * kStage16, n > 0 ? 1u : 0u);  // dK += dS^T Q
          commit(bar_ld_empty + st);
          if (n + 2 < N) {                                                  // S^T(n+2) into the buffer P^T(n), dS^T(n) just left:
            ok = mbar_wait(bar_ld_full + st2, ph2, a.status);               // it heads the next step's dependency chain, so it
            if (!ok) return;                                                // goes ahead of dQ^T(n), which only feeds the drain
            clear_stage_tail(st2);
            tc_fence_after();
            gemm_st(sbuf, dK_k, dQ_k0 + st2 * kStage16);
            commit(bar_s_full + b_);
          }
          gemm_dq(dpbuf, dDS0 + b_ * kDS16);                                // dQ^T = K^T dS^T over the consumed dP^T(n)
          commit(bar_dq_full + b_);
          // advance the bookkeeping to step n+1
          st = st1; st1 = st2;
          if (++st2 == NST) { st2 = 0; ph2 ^= 1; }
          if (b_ == 1) par ^= 1;
        };
        for (int n = 0; n < N && ok; n += 2) {
          body(n, std::integral_constant<int, 0>{});
          if (n + 1 < N && ok) body(n + 1, std::integral_constant<int, 1>{});
        }
        commit(bar_done);
      }
    }
  } else if (warp < 12) {
    setmaxnreg_inc<160>();
    {
      // ======== two compute warpgroups, each takes 32 of the 64 query columns of every step: P^T and dS^T, one
      // KV row per thread.  Inside the 64-column S^T buffer a warpgroup only ever writes into the 32 columns
      // it reads: P^T (bf16 pairs) into the first 16 of them, dS^T into the last 16.
      const int wg = (warp - 4) >> 2;        // query columns [32 wg, 32 wg + 32) of every step
      const int r = (warp & 3) * 32 + lane;  // KV row = TMEM lane
      const uint32_t t_lane = tmem_base + ((uint32_t)((warp & 3) * 32) << 16);
      const int kcol = k0 + r;               // key index of this thread
      const long long kpos = (long long)kcol - off;  // first causal query of this key
      const float2 sc2 = make_float2(a.scale_log2, a.scale_log2);
      int st = 0, t_in = tq0;                // stage and position in I_h(j) of the next step
      uint32_t ph_l = 0, par = 0;
      for (int n = 0; n < N && ok; ++n) {
        const int b_ = n & 1;
        const uint32_t sbuf = t_lane + cS0 + b_ * 64 + wg * 32, dpbuf = t_lane + cDP0 + b_ * 64 + wg * 32;
        uint8_t* ds_row = sDS + b_ * SM::kDS + r * 128;
        const int i = cowa_bwd_tile_at(rg, t_in);
        const int q0 = i * BQS;
        const bool full = cowa_tile_full(w, q0, BQS, k0, BKV, off, Nq, Nk);
        uint32_t mk = 0xFFFFFFFFu;
        if (!full) {
          const long long qend = Nq - 1;
          const long long base = q0 + wg * 32;
          uint32_t m = interval_bits32(kpos, min(kpos + w.n - 1, qend), base);
          if (w.l > 0)
            m |= interval_bits32(kpos + w.n + w.g, min(kpos + (long long)w.n + w.g + w.l - 1, qend), base);
          if (kcol < w.s) m |= interval_bits32(kpos, qend, base);
          mk = kcol < Nk ? m : 0u;
        }
        const float4* nlse4 = reinterpret_cast<const float4*>(sVec + st * 128 + wg * 32);  // -LSE log2(e), then -Delta
        const float4* ndlt4 = nlse4 + 16;
        ok = mbar_wait(bar_ld_full + st, ph_l, a.status);
        ok = ok && mbar_wait(bar_s_full + b_, par, a.status);
        if (!ok) break;
        tc_fence_after();
        float p[32];
        {
          uint32_t sr[32], pk[16];
          tmem_ld32(sbuf, sr);
          tmem_wait_ld();
#pragma unroll
          for (int e = 0; e < 32; e += 4) {
            const float4 nl = nlse4[e / 4];
            const float2 x = fma2(make_float2(__uint_as_float(sr[e]), __uint_as_float(sr[e + 1])), sc2, make_float2(nl.x, nl.y));
            const float2 y = fma2(make_float2(__uint_as_float(sr[e + 2]), __uint_as_float(sr[e + 3])), sc2, make_float2(nl.z, nl.w));
            p[e] = ex2(x.x);
            p[e + 1] = ex2(x.y);
            p[e + 2] = ex2(y.x);
            p[e + 3] = ex2(y.y);
          }
          if (!full) {
#pragma unroll
            for (int e = 0; e < 32; ++e)
              if (!((mk >> e) & 1u)) p[e] = 0.f;
          }
#pragma unroll
          for (int e = 0; e < 32; e += 2) pk[e / 2] = pack_bf16(p[e], p[e + 1]);
          tmem_st16(sbuf, pk);  // P^T: this warpgroup's 32 queries as 16 bf16 pairs
        }
        tmem_wait_st();
        tc_fence_before();
        mbar_arrive(bar_p_ready + b_);

        ok = mbar_wait(bar_dp_full + b_, par, a.status);
        if (!ok) break;
        tc_fence_after();
        {
          uint32_t dr[32], dsp[16];
          tmem_ld32(dpbuf, dr);
          tmem_wait_ld();
#pragma unroll
          for (int e = 0; e < 32; e += 4) {
            const float4 nd = ndlt4[e / 4];
            const float2 y = mul2(make_float2(p[e], p[e + 1]),
                                  add2(make_float2(__uint_as_float(dr[e]), __uint_as_float(dr[e + 1])), make_float2(nd.x, nd.y)));
            const float2 z = mul2(make_float2(p[e + 2], p[e + 3]),
                                  add2(make_float2(__uint_as_float(dr[e + 2]), __uint_as_float(dr[e + 3])), make_float2(nd.z, nd.w)));
            dsp[e / 2] = pack_bf16(y.x, y.y);
            dsp[e / 2 + 1] = pack_bf16(z.x, z.y);
          }
          tmem_st16(sbuf + 16, dsp);  // dS^T beside P^T
          // dS^T also to shared memory (row r = 128 B = 8 chunks, 128B swizzle) for the dQ^T product
#pragma unroll
          for (int ch = 0; ch < 4; ++ch)
            *reinterpret_cast<uint4*>(ds_row + (((wg * 4 + ch) ^ (r & 7)) << 4)) =
                make_uint4(dsp[ch * 4], dsp[ch * 4 + 1], dsp[ch * 4 + 2], dsp[ch * 4 + 3]);
        }
        tmem_wait_st();
        tc_fence_before();
        fence_proxy_async_smem();
        mbar_arrive(bar_ds_ready + b_);
        if (b_) par ^= 1;
        if (++st == NST) { st = 0; ph_l ^= 1; }
        if (++t_in == cnt) t_in = 0;
      }
      if (wg == 0) store_grad(true);
    }
  } else {
    setmaxnreg_dec<112>();
    {
      // ======== dQ drain warpgroup: one d column of dQ^T per thread; TMEM -> shared -> bulk reduce-add ========
      const int d = (warp & 3) * 32 + lane;
      const uint32_t t_lane = tmem_base + ((uint32_t)((warp & 3) * 32) << 16);
      const bool issuer = (d == 0);
      int g = g0, t_in = tq0;
      for (int n = 0; n < N && ok; ++n) {
        const int i = cowa_bwd_tile_at(rg, t_in);
        const int bhq = bhq0 + g, q0 = i * BQS;
        if (++t_in == cnt) { t_in = 0; ++g; }
        ok = mbar_wait(bar_dq_full + (n & 1), (n >> 1) & 1, a.status);
        if (!ok) break;
        tc_fence_after();
        uint32_t v[2][32];
        tmem_ld32(t_lane + cDP0 + (n & 1) * 64, v[0]);
        tmem_ld32(t_lane + cDP0 + (n & 1) * 64 + 32, v[1]);
        tmem_wait_ld();
        tc_fence_before();
        mbar_arrive(bar_dq_free + (n & 1));
#pragma unroll
        for (int hf = 0; hf < 2; ++hf) {
          float* stage = sDQ + hf * (SM::kDQ / 4);
          if (issuer) tma_wait_group_read<1>();  // the reduction issued from this tile one step ago has read it
          wg_sync(3);
          if (d < D) {
            if (a.dq_fixed) {
              // Rounded to integers on the FMA and integer pipes (the conversion instruction runs at the rate of the
              // exponentials and competed with them: one KV head of 20001 tokens 942 / 880 thousand clocks): x = 2^16 h + l
              // with h = rint(x / 2^16), |l| <= 2^15, both exact; adding 1.5 * 2^23 leaves an integer in the low mantissa
              // bits, and shifting the first sum by 16 drops its exponent.  Same integers as __float2int_rn.
              const float2 fx2 = make_float2(a.scale * kDqFixedOne, a.scale * kDqFixedOne);
              auto c2 = [](float c_) { return make_float2(c_, c_); };
              float worst = 0.f;
#pragma unroll
              for (int c = 0; c < 32; c += 2) {
                const float2 x = mul2(make_float2(__uint_as_float(v[hf][c]), __uint_as_float(v[hf][c + 1])), fx2);
                worst = max_nan(worst, max_nan(fabsf(x.x), fabsf(x.y)));
                const float2 th = fma2(x, c2(1.f / 65536.f), c2(12582912.f));
                const float2 l = fma2(add2(th, c2(-12582912.f)), c2(-65536.f), x);
                const float2 tl = add2(l, c2(12582912.f));
                int* dst = reinterpret_cast<int*>(stage) + c * D + d;
                dst[0] = (__float_as_int(th.x) << 16) + (__float_as_int(tl.x) - 0x4B400000);
                dst[D] = (__float_as_int(th.y) << 16) + (__float_as_int(tl.y) - 0x4B400000);
              }
              if (!(worst < 2147483520.f)) atomicOr(a.status, (unsigned)COWA_DEV_DQ_RANGE);  // would not fit 32 bits (or NaN)
            } else {
#pragma unroll
              for (int c = 0; c < 32; ++c) stage[c * D + d] = __uint_as_float(v[hf][c]) * a.scale;
            }
          }
          fence_proxy_async_smem();
          wg_sync(3);
          if (issuer) {
            // 32 query rows of the accumulator are one contiguous range (rows are D floats, padded row space)
            void* gdst = a.dq_acc + (((size_t)bhq * vec_stride + pbase + q0 + hf * 32) * D);
            if (a.dq_fixed) bulk_reduce_add_s32(gdst, stage, 32 * D * 4);
            else bulk_reduce_add_f32(gdst, stage, 32 * D * 4);
            tma_commit_group();
          }
        }
      }
      if (issuer) tma_wait_group<0>();
      store_grad(false);
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    __syncwarp();
    tmem_dealloc(tmem_base, TMEM_COLS);
  }
}

// delta = -rowsum(O * dO), lse2 = -LSE * log2(e); rows in [T, Tpad) get lse2 = -inf, delta = 0.  The same threads zero
// the fp32 dQ accumulator (as a memset before it that was a pass of its own: 32K 190 us for both, 164 us so).
template <int D>
__global__ void cowa_bwd_preprocess_kernel(const __nv_bfloat16* __restrict__ o, const __nv_bfloat16* __restrict__ d_o,
                                           const float* __restrict__ lse, float* __restrict__ lse2,
                                           float* __restrict__ delta, float* __restrict__ acc, int T, int Tpad,
                                           long long BH, int H, CowaStrides so) {
  constexpr int TPR = D / 8;  // threads per row (16 bytes each)
  const long long gid = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const long long row = gid / TPR;
  const int part = (int)(gid % TPR);
  if (row >= BH * Tpad) return;
  const long long bh = row / Tpad;
  const int t = (int)(row % Tpad);
  float4* z = reinterpret_cast<float4*>(acc + (size_t)row * D + part * 8);
  z[0] = z[1] = make_float4(0.f, 0.f, 0.f, 0.f);
  float s = 0.f;
  if (t < T) {
    const size_t base = (size_t)(bh / H) * so.b + (size_t)(bh % H) * so.h + (size_t)t * so.t + part * 8;
    const uint4 x = *reinterpret_cast<const uint4*>(o + base);
    const uint4 y = *reinterpret_cast<const uint4*>(d_o + base);
    const uint32_t xs[4] = {x.x, x.y, x.z, x.w}, ys[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      s = fmaf(__uint_as_float(xs[i] << 16), __uint_as_float(ys[i] << 16), s);
      s = fmaf(__uint_as_float(xs[i] & 0xffff0000u), __uint_as_float(ys[i] & 0xffff0000u), s);
    }
  }
#pragma unroll
  for (int o_ = TPR / 2; o_ > 0; o_ >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o_);
  if (part == 0) {
    delta[row] = -s;
    lse2[row] = t < T ? lse[(size_t)bh * T + t] * -1.4426950408889634f : -INFINITY;
  }
}

// Packed batches.  One block per (64-row chunk of the padded row space, QO head): -Delta and -LSE * log2(e)
// of the chunk's rows (padding rows: -inf, 0), read from the packed tensors.
template <int D>
__global__ void cowa_bwd_preprocess_varlen_kernel(const __nv_bfloat16* __restrict__ o,
                                                  const __nv_bfloat16* __restrict__ d_o,
                                                  const float* __restrict__ lse, float* __restrict__ lse2,
                                                  float* __restrict__ delta, float* __restrict__ acc,
                                                  const int* __restrict__ cu, int B, int total, int Tpad,
                                                  unsigned int* status) {
  constexpr int TPR = D / 8;  // threads per row (16 bytes each)
  const int chunk = blockIdx.x, h = blockIdx.y;
  const int r = threadIdx.x / TPR, part = threadIdx.x % TPR;
  int b, lc, nch, pb;
  if (chunk == 0 && h == 0 && threadIdx.x < 32 && varlen_locate(cu, B, Tpad / BQS, BQS, BQS, &b, &lc, &nch, &pb) &&
      threadIdx.x == 0)
    atomicOr(status, (unsigned)COWA_DEV_BAD_SEQLENS);  // more chunks than the row space holds: see fits
  const bool in = varlen_locate(cu, B, chunk, BQS, BQS, &b, &lc, &nch, &pb);
  const int t = lc * BQS + r;  // row inside the sequence
  const int rbase = in ? cu[b] : 0;
  const bool valid = in && t < cu[b + 1] - rbase && rbase >= 0 && rbase + t < total;
  float4* z = reinterpret_cast<float4*>(acc + ((size_t)h * Tpad + (size_t)chunk * BQS + r) * D + part * 8);
  z[0] = z[1] = make_float4(0.f, 0.f, 0.f, 0.f);
  float s = 0.f;
  if (valid) {
    const size_t base = ((size_t)h * total + rbase + t) * D + part * 8;
    const uint4 x = *reinterpret_cast<const uint4*>(o + base);
    const uint4 y = *reinterpret_cast<const uint4*>(d_o + base);
    const uint32_t xs[4] = {x.x, x.y, x.z, x.w}, ys[4] = {y.x, y.y, y.z, y.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      s = fmaf(__uint_as_float(xs[i] << 16), __uint_as_float(ys[i] << 16), s);
      s = fmaf(__uint_as_float(xs[i] & 0xffff0000u), __uint_as_float(ys[i] & 0xffff0000u), s);
    }
  }
#pragma unroll
  for (int o_ = TPR / 2; o_ > 0; o_ >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o_);
  if (part == 0) {
    const size_t row = (size_t)h * Tpad + (size_t)chunk * BQS + r;  // chunks are laid out in order: pb == chunk * BQS
    delta[row] = -s;
    lse2[row] = valid ? lse[(size_t)h * total + rbase + t] * -1.4426950408889634f : -INFINITY;
  }
}

// 8 elements of the dQ accumulator (fp32, or 32-bit integers in units of 2^-18) -> bf16
__device__ __forceinline__ uint4 dq_bf16(const float4* src, int fixed, unsigned int* status) {
  float4 x = src[0], y = src[1];
  if (fixed) {
    const float u = 1.f / kDqFixedOne;
    x = make_float4(__float_as_int(x.x) * u, __float_as_int(x.y) * u, __float_as_int(x.z) * u, __float_as_int(x.w) * u);
    y = make_float4(__float_as_int(y.x) * u, __float_as_int(y.y) * u, __float_as_int(y.z) * u, __float_as_int(y.w) * u);
    // half of the representable range: a total that wrapped around lands out here in most cases
    const float big = fmaxf(fmaxf(fmaxf(fabsf(x.x), fabsf(x.y)), fmaxf(fabsf(x.z), fabsf(x.w))),
                            fmaxf(fmaxf(fabsf(y.x), fabsf(y.y)), fmaxf(fabsf(y.z), fabsf(y.w))));
    if (big >= 4096.f) atomicOr(status, (unsigned)COWA_DEV_DQ_RANGE);
  }
  return make_uint4(pack_bf16(x.x, x.y), pack_bf16(x.z, x.w), pack_bf16(y.x, y.y), pack_bf16(y.z, y.w));
}

// The dQ accumulator to bf16.  Batched: 8 elements a thread; packed: one 64-row chunk of the padded row space and one head a
// block, into the packed rows.  (One kernel with the sum of partial dK, dV needs 46 registers and lost occupancy: 137
// instead of 112 us at 32K.)
template <int D, bool VARLEN>
__global__ void __launch_bounds__(VARLEN ? BQS * (D / 8) : 256)
cowa_bwd_convert_dq_kernel(const float* __restrict__ acc, __nv_bfloat16* __restrict__ dq, const int* __restrict__ cu, int B,
                           int T, int Tpad, long long BH, int H, int fixed, CowaStrides sq, unsigned int* status) {
  constexpr int TPR = D / 8;  // threads per row (16 bytes of bf16 each)
  const int part = threadIdx.x % TPR;
  if constexpr (!VARLEN) {
    const long long row = ((long long)blockIdx.x * blockDim.x + threadIdx.x) / TPR;
    if (row >= BH * T) return;
    const long long bh = row / T;
    const int t = (int)(row % T);
    const uint4 v = dq_bf16(reinterpret_cast<const float4*>(acc + ((size_t)bh * Tpad + t) * D + part * 8), fixed, status);
    *reinterpret_cast<uint4*>(dq + (size_t)(bh / H) * sq.b + (size_t)(bh % H) * sq.h + (size_t)t * sq.t + part * 8) = v;
  } else {
    const int chunk = blockIdx.x, h = blockIdx.y, r = threadIdx.x / TPR;
    int b, lc, nch, pb;
    if (!varlen_locate(cu, B, chunk, BQS, BQS, &b, &lc, &nch, &pb)) return;
    const int t = lc * BQS + r;
    const int rbase = cu[b];
    if (t >= cu[b + 1] - rbase || rbase < 0 || rbase + t >= T) return;
    const uint4 v = dq_bf16(reinterpret_cast<const float4*>(acc + ((size_t)h * Tpad + (size_t)chunk * BQS + r) * D + part * 8),
                            fixed, status);
    *reinterpret_cast<uint4*>(dq + ((size_t)h * T + rbase + t) * D + part * 8) = v;
  }
}

// Partial dK (blockIdx.y = 0) and dV (1) of the shared tiles, added in slot order, to bf16.
template <int D, bool VARLEN>
__global__ void __launch_bounds__(256)
cowa_bwd_reduce_dkv_kernel(const __grid_constant__ BwdArgs a, CowaStrides sk, CowaStrides sv) {
  constexpr int TPR = D / 8, ROWS = 256 / TPR;  // threads per row (16 bytes of bf16 each), rows per block
  const int part = threadIdx.x % TPR;
  int q = blockIdx.x / (BKV / ROWS), c = 0, slot = 0;
  const int r = blockIdx.x % (BKV / ROWS) * ROWS + threadIdx.x / TPR;
  for (; c < 2; ++c) {
    if (a.cls_parts[c] == 1) continue;
    if (q < a.cls_tiles[c]) break;
    q -= a.cls_tiles[c];
    slot += a.cls_tiles[c] * a.cls_parts[c];
  }
  const int parts = a.cls_parts[c];
  TileAt at;
  if (!locate_tile<VARLEN>(a, c, q, at)) return;
  int Nk = a.Nk, rbase = 0;
  if constexpr (VARLEN) {
    rbase = a.cu[at.b];
    Nk = a.cu[at.b + 1] - rbase;
    if (rbase < 0 || rbase + Nk > a.total) return;
  }
  const int t = at.j * BKV + r;
  if (t >= Nk) return;
  const int m = blockIdx.y;
  // the slots hold a row's 16-byte chunks permuted
  const float* src = a.dkv_part + ((size_t)(slot + q * parts) * 2 + m) * (BKV * D) + (size_t)r * D;
  const int c0 = ((part * 2) ^ (r & 7)) * 4, c1 = ((part * 2 + 1) ^ (r & 7)) * 4;
  float4 x = make_float4(0.f, 0.f, 0.f, 0.f), y = x;
#pragma unroll 4
  for (int i = 0; i < parts; ++i) {
    const float4 u = *reinterpret_cast<const float4*>(src + (size_t)i * 2 * (BKV * D) + c0);
    const float4 v = *reinterpret_cast<const float4*>(src + (size_t)i * 2 * (BKV * D) + c1);
    x.x += u.x; x.y += u.y; x.z += u.z; x.w += u.w;
    y.x += v.x; y.y += v.y; y.z += v.z; y.w += v.w;
  }
  const size_t o = VARLEN ? ((size_t)at.hk * a.total + rbase + t) * D
                 : m == 0 ? (size_t)at.b * sk.b + (size_t)at.hk * sk.h + (size_t)t * sk.t
                          : (size_t)at.b * sv.b + (size_t)at.hk * sv.h + (size_t)t * sv.t;
  *reinterpret_cast<uint4*>((m == 0 ? a.dk : a.dv) + o + part * 8) =
      make_uint4(pack_bf16(x.x, x.y), pack_bf16(x.z, x.w), pack_bf16(y.x, y.y), pack_bf16(y.z, y.w));
}

// How the KV tiles are shared among blocks.  A tile whose block takes the whole GQA group keeps dK, dV in TMEM; a shared
// tile costs every block a prologue and 128 KB of fp32 partial sums (D = 128), about four steps' worth of time, so tiles
// are shared only where whole ones leave SMs idle:
//   sink tiles, visited by every query tile, when one is longer than 3/4 of an SM's share of the work: thirds of a share;
//   all tiles when there are at most two per SM: fifths of a share, four steps at least;
//   the last tile per SM when there are at most eight: quarters, so that the last wave ends together.
// Main kernel, 1000 clocks, whole heads of a group spread / this: 2 x 8K, 16 heads 1147 / 1070; one KV head of 20001 tokens
// 1021 / 983; 1K, 4 heads 58 / 34.
struct BwdPlan {
  int sink_tiles;  // per sequence and head
  int tiles[3], parts[3];
  long long slots() const {
    long long n = 0;
    for (int c = 0; c < 3; ++c)
      if (parts[c] > 1) n += (long long)tiles[c] * parts[c];
    return n;
  }
  long long blocks() const {
    long long n = 0;
    for (int c = 0; c < 3; ++c) n += (long long)tiles[c] * parts[c];
    return n;
  }
};

// `rest` tiles behind the sink tiles, `avg` steps each; share: an SM's steps
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

BwdPlan bwd_plan(int B, int Nq, int Nk, int Hkv, int G, const CowaHeadWindows& hw) {
  BwdPlan pl;
  const int nKV = (Nk + BKV - 1) / BKV, sms = cowa::sm_count();
  pl.sink_tiles = 0;
  for (int h = 0; h < Hkv; ++h) pl.sink_tiles = std::max(pl.sink_tiles, (std::min(hw.w[h].s, Nk) + BKV - 1) / BKV);
  long long total = 0, sinks = 0, longest = 0, longest_sink = 0;
  for (int h = 0; h < Hkv; ++h)
    for (int j = 0; j < nKV; ++j) {
      CowaRange rg[2];
      const int k0 = j * BKV, k1 = std::min(k0 + BKV, Nk) - 1;
      cowa_bwd_ranges(hw.w[h], k0, k1, Nk - Nq, Nq, BQS, rg);
      const long long cnt = (long long)(cowa_range_len(rg[0]) + cowa_range_len(rg[1])) * G;
      total += cnt;
      longest = std::max(longest, cnt);
      if (j < pl.sink_tiles) { sinks += cnt; longest_sink = std::max(longest_sink, cnt); }
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

template <int D, bool VARLEN>
void launch_reduce(const BwdArgs& a, const BwdPlan& pl, const CowaStrides& sk, const CowaStrides& sv, cudaStream_t st) {
  long long shared = 0;
  for (int c = 0; c < 3; ++c)
    if (pl.parts[c] > 1) shared += pl.tiles[c];
  if (shared > 0)
    cowa_bwd_reduce_dkv_kernel<D, VARLEN><<<dim3((unsigned)(shared * (BKV * (D / 8) / 256)), 2), 256, 0, st>>>(a, sk, sv);
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
  CUtensorMap mq, mk, mv, mdo, mdk, mdv;
  if ((rc = cowa::make_tensor_map(&mq, q, cowa::MapType::BF16, D, T, Hq, B, sq, 64, BQS))) return rc;
  if ((rc = cowa::make_tensor_map(&mdo, d_o, cowa::MapType::BF16, D, T, Hq, B, so, 64, BQS))) return rc;
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
  for (int c = 0; c < 3; ++c) { a.cls_tiles[c] = pl.tiles[c]; a.cls_parts[c] = pl.parts[c]; }
  a.dq_fixed = p->deterministic ? 1 : 0;
  a.dkv_part = dkv_part;
  a.cu = nullptr; a.dk = static_cast<__nv_bfloat16*>(dk); a.dv = static_cast<__nv_bfloat16*>(dv); a.total = 0; a.tiles_bound = 0;
  a.sink = 0; a.local = 0; a.hkv_global = 0; a.hkv_offset = 0; a.full_attn = 0; a.explicit_windows = 0;
  if (pl.blocks() > 0x7FFFFFFFll || (long long)Nq / BQS * a.G * 32 > 0x7FFFFFFFll) return COWA_ERR_UNSUPPORTED;
  COWA_CUDA_TRY(cudaFuncSetAttribute(cowa_bwd_kernel<D, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     BwdSmem<D>::kBytes));
  {
    const long long threads = BH * Tpad * (D / 8);
    cowa_bwd_preprocess_kernel<D><<<(unsigned)((threads + 255) / 256), 256, 0, st>>>(
        static_cast<const __nv_bfloat16*>(o), static_cast<const __nv_bfloat16*>(d_o), lse, lse2, delta, dq_acc,
        T, Tpad, BH, Hq, so);
    COWA_CUDA_TRY(cudaGetLastError());
  }
  if (p->bwd_main_start_event) COWA_CUDA_TRY(cudaEventRecord(static_cast<cudaEvent_t>(p->bwd_main_start_event), st));
  cowa_bwd_kernel<D, false><<<(unsigned)pl.blocks(), 512, BwdSmem<D>::kBytes, st>>>(mq, mk, mv, mdo, mdk, mdv, a);
  COWA_CUDA_TRY(cudaGetLastError());
  if (p->bwd_main_stop_event) COWA_CUDA_TRY(cudaEventRecord(static_cast<cudaEvent_t>(p->bwd_main_stop_event), st));
  launch_reduce<D, false>(a, pl, sk, sv, st);
  COWA_CUDA_TRY(cudaGetLastError());
  cowa_bwd_convert_dq_kernel<D, false><<<(unsigned)((BH * T * (D / 8) + 255) / 256), 256, 0, st>>>(
      dq_acc, static_cast<__nv_bfloat16*>(dq), nullptr, B, T, Tpad, BH, Hq, a.dq_fixed, sq, a.status);
  COWA_CUDA_TRY(cudaGetLastError());
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
  CUtensorMap mq, mk, mv, mdo, mdk, mdv;
  int rc;
  const CowaStrides sq = packed_strides(Hq, total, D), sk = packed_strides(Hkv, total, D);
  if ((rc = cowa::make_tensor_map(&mq, q, cowa::MapType::BF16, D, total, Hq, 1, sq, 64, BQS))) return rc;
  if ((rc = cowa::make_tensor_map(&mdo, d_o, cowa::MapType::BF16, D, total, Hq, 1, sq, 64, BQS))) return rc;
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
  for (int c = 0; c < 3; ++c) { a.cls_tiles[c] = pl.tiles[c]; a.cls_parts[c] = pl.parts[c]; }
  a.dq_fixed = p->deterministic ? 1 : 0;
  a.dkv_part = delta + (size_t)Hq * Tpad;
  a.cu = cu; a.dk = static_cast<__nv_bfloat16*>(dk); a.dv = static_cast<__nv_bfloat16*>(dv);
  a.total = total; a.tiles_bound = total / BKV + B;
  a.sink = p->sink; a.local = p->local;
  a.hkv_global = p->hkv_global > 0 ? p->hkv_global : Hkv;
  a.hkv_offset = p->hkv_offset; a.full_attn = p->full_attn; a.explicit_windows = p->windows != nullptr;
  if (pl.blocks() > 0x7FFFFFFFll || (long long)total / BQS * a.G * 32 > 0x7FFFFFFFll) return COWA_ERR_UNSUPPORTED;
  COWA_CUDA_TRY(cudaFuncSetAttribute(cowa_bwd_kernel<D, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     BwdSmem<D>::kBytes));
  const dim3 chunks(Tpad / BQS, Hq);
  cowa_bwd_preprocess_varlen_kernel<D><<<chunks, BQS * (D / 8), 0, st>>>(
      static_cast<const __nv_bfloat16*>(o), static_cast<const __nv_bfloat16*>(d_o), lse, lse2, delta, dq_acc,
      cu, B, total, Tpad, a.status);
  COWA_CUDA_TRY(cudaGetLastError());
  if (p->bwd_main_start_event) COWA_CUDA_TRY(cudaEventRecord(static_cast<cudaEvent_t>(p->bwd_main_start_event), st));
  cowa_bwd_kernel<D, true><<<(unsigned)pl.blocks(), 512, BwdSmem<D>::kBytes, st>>>(mq, mk, mv, mdo, mdk, mdv, a);
  COWA_CUDA_TRY(cudaGetLastError());
  if (p->bwd_main_stop_event) COWA_CUDA_TRY(cudaEventRecord(static_cast<cudaEvent_t>(p->bwd_main_stop_event), st));
  launch_reduce<D, true>(a, pl, sk, sk, st);
  COWA_CUDA_TRY(cudaGetLastError());
  cowa_bwd_convert_dq_kernel<D, true><<<chunks, BQS * (D / 8), 0, st>>>(dq_acc, static_cast<__nv_bfloat16*>(dq), cu, B, total,
                                                                        Tpad, 0, Hq, a.dq_fixed, sq, a.status);
  COWA_CUDA_TRY(cudaGetLastError());
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
  return ws_bytes(B, Nq, Hq, D, bwd_plan(B, Nq, Nk, Hkv, Hq / Hkv, hw));
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
  const BwdPlan pl = bwd_plan(B, Nq, Nk, Hkv, Hq / Hkv, hw);
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
