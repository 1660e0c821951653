// CoWindow Attention forward (Algorithm 1) for sm_100a: two QO heads of a GQA group per block.
//
// One block per SM at a time, each taking over further blocks of the grid (cluster launch control).  A work item is (batch, pair of QO
// heads that share a KV head, 128-row QO tile);
// both heads visit the same KV tiles J_h(i), so one pass over K and V serves 256 query rows.  A step takes two
// visited 64-key tiles (not necessarily neighbours) as one 128-key operand: S at N = 128 runs at the full tensor
// rate (512 clocks; as two products of 64 keys 768).  Warps:
//   warps 0-3, 4-7  softmax of head 0 / head 1: one query row per thread; then O / l and LSE
//   warp 8          TMA producer: Q of both heads, then K and V of every step through four 32 KB slots; works out the
//                   items' geometry one item ahead
//   warp 9          MMA issuer, per step:  O_0 += P_0 V | S_0' = Q_0 K' | O_1 += P_1 V | S_1' = Q_1 K'
// While the tensor pipe works for one head, the other head's warps do their softmax, so the two alternate.
// P is handed over in two halves: O += P V starts on the first while the second is still being exponentiated.
// P overwrites S in TMEM; S_0 (128 columns), S_1, O_0, O_1 fill all 512 columns.
// As in the one-head kernel the running max only advances when it grows by more than 2^8; S of a step completes
// after O += P V of the step before it (same issue order), so the rare rescale needs no further wait.
// The next item's Q, K and V are fetched, and its first S computed, while the softmax warps still write out O.
//
// What bounds it: per step and pair of heads the tensor pipe needs 2048 clocks and the exponentials 2048 of the
// special-function unit (1792 with one pair in eight on the FMA pipe); a step takes about 3150, the chain of one
// head (S landed 900, load 100, row max 300, exponentials 1400, hand-over 150, with one warp per scheduler and
// head to cover it) at 1.7 GHz; long calls run at the power limit below that.
#include "cowa_fwd.h"

#include <algorithm>
#include <atomic>

using namespace cowa_ptx;

namespace {

constexpr int BQ = 128, BK = 64, BS = 2 * BK;  // query rows per tile, keys per visited tile, keys per step
constexpr int kSplitQ = 1;  // O += P V starts once the 32-key groups 0 .. kSplitQ of P are in place
constexpr int kPairThreads = 384;  // warps 10, 11 only make the control warpgroup whole
constexpr int kItemReaders = 9;  // warps that read a published work item: softmax 8, MMA 1

// 2^x of a pair on the FMA and integer pipes: x = n + f with n = rint(x), |f| <= 1/2, 2^f by the polynomial of
// degree 6 with the least largest relative error on that interval (fitted by reweighted least squares: 1.9e-9, in
// fp32 8e-8, against 2 ulp of ex2.approx), times 2^n.  x is held at -127 from below, where the
// exponent word of 2^n is 0: a masked score (-inf) weighs exactly 0, as ex2.approx gives it; NaN stays NaN.
__device__ __forceinline__ float2 exp2_fma(float2 x) {
  auto c2 = [](float c) { return make_float2(c, c); };
  x.x = max_nan(x.x, -127.f); x.y = max_nan(x.y, -127.f);
  const float2 t = add2(x, c2(12582912.f));                        // 1.5 * 2^23: n in the low mantissa bits
  const float2 f = fma2(add2(t, c2(-12582912.f)), c2(-1.f), x);
  float2 p = fma2(c2(1.53458118e-4f), f, c2(1.33999312e-3f));
  p = fma2(p, f, c2(9.61848896e-3f));
  p = fma2(p, f, c2(5.55032878e-2f));
  p = fma2(p, f, c2(2.40226469e-1f));
  p = fma2(p, f, c2(6.93147206e-1f));
  p = fma2(p, f, c2(1.f));
  return mul2(p, make_float2(__uint_as_float((__float_as_uint(t.x) << 23) + 0x3F800000u),
                             __uint_as_float((__float_as_uint(t.y) << 23) + 0x3F800000u)));
}

template <int D>
struct PairSmem {
  static constexpr int kQ = BQ * D * 2;    // Q tile of one head
  static constexpr int kKV = BS * D * 2;   // K or V operand of one step
  static constexpr int kOut = BQ * 128;    // one 64-column slab of an O tile on its way out
  static constexpr int oQ = 0, oK = 2 * kQ, oV = oK + 2 * kKV, oOut = oV + 2 * kKV, oBar = oOut + 2 * kOut;
  static constexpr int oNext = oBar + 240;           // the next item's number, as the hardware answers
  static constexpr int oItem = oBar + 256;           // two work items
  static constexpr int kBytes = oItem + 256 + 1024;  // + alignment slack
};
static_assert(PairSmem<128>::kBytes <= 232448, "shared memory of a block");

// One work item: where its rows lie, which KV tiles it visits and which of them need no mask.  The TMA warp works
// it out one item ahead and leaves it in shared memory for the other warps.
struct PairItem {
  int b, bt, h0, hk, Nq, Nk, qbase, kbase, q0, off;
  CowaWin w;
  CowaRange rg[3];
  int f_lo[3], f_hi[3];  // unmasked tiles: one interval per range (see cowa_fwd_kernel)
  int t0, nt;            // visited 64-key tiles of this block: t0 .. t0 + nt - 1 of the list; nt = 0: no more items
  int work;              // split items: 0 when there is nothing to write at all
};
static_assert(sizeof(PairItem) <= 128, "slot of a published item");
static_assert(4 * PairSmem<128>::kKV >= 2 * BQ * 128 * 4, "fp32 O of both heads fits the K and V slots");

// false: no item of this number (packed batches: the count is an upper bound; it.b = -1) or malformed offsets
template <bool VARLEN>
__device__ __forceinline__ bool locate_item(const FwdArgs& a, int idx, PairItem& it) {
  const int PG = a.G >> 1;
  const int gp = idx % PG; idx /= PG;
  it.hk = idx % a.Hkv; idx /= a.Hkv;
  it.h0 = it.hk * a.G + 2 * gp;
  int i;
  it.w = a.wins.w[it.hk];
  if constexpr (!VARLEN) {
    it.b = idx % a.B; idx /= a.B;
    i = (a.Nq + BQ - 1) / BQ - 1 - idx;  // heaviest tiles first
    it.Nq = a.Nq; it.Nk = a.Nk; it.qbase = 0; it.kbase = 0; it.bt = it.b;
  } else {
    int lt, nts, pb;
    if (a.longest_first ? !varlen_locate_longest(a.cu_q, a.cu_k, a.B, idx, BQ, 1, 0, &it.b, &lt, &nts)
                        : !varlen_locate(a.cu_q, a.B, idx, BQ, 0, &it.b, &lt, &nts, &pb)) {
      it.b = -1;
      return false;
    }
    i = nts - 1 - lt;
    it.qbase = a.cu_q[it.b]; it.Nq = a.cu_q[it.b + 1] - it.qbase;
    it.kbase = a.cu_k[it.b]; it.Nk = a.cu_k[it.b + 1] - it.kbase;
    it.bt = 0;
    if (it.Nq > it.Nk || it.qbase < 0 || it.kbase < 0 || it.qbase + it.Nq > a.total_q || it.kbase + it.Nk > a.total_k) {
      if ((threadIdx.x & 31) == 0) atomicOr(a.status, (unsigned)COWA_DEV_BAD_SEQLENS);
      return false;
    }
    if (a.full_attn) { it.w.s = 0; it.w.n = it.Nk; it.w.g = 0; it.w.l = 0; }
    else if (!a.explicit_windows) it.w = cowa_default_window(it.Nk, a.hkv_global, a.hkv_offset + it.hk, a.sink, a.local);
  }
  const CowaWin w = it.w;
  it.off = it.Nk - it.Nq;
  it.q0 = i * BQ;
  cowa_fwd_ranges(w, it.q0, min(it.q0 + BQ, it.Nq) - 1, it.off, it.Nk, BK, it.rg);
  it.t0 = 0;
  it.nt = cowa_range_len(it.rg[0]) + cowa_range_len(it.rg[1]) + cowa_range_len(it.rg[2]);
  it.work = it.nt;
#pragma unroll
  for (int q = 0; q < 3; ++q) { it.f_lo[q] = 1; it.f_hi[q] = 0; }
  if (it.q0 + BQ <= it.Nq) {
    auto fdiv = [](long long v) -> int { return (int)(v >> 6); };  // floor of v / BK
    static_assert(BK == 64, "shift in fdiv");
    const long long p0 = (long long)it.q0 + it.off, p1 = p0 + BQ - 1;
    const int causal_hi = fdiv(p0 - (BK - 1));
    it.f_lo[0] = fdiv(p1 - w.n) + 1; it.f_hi[0] = causal_hi;
    if (w.l > 0) {
      it.f_lo[1] = fdiv(p1 - ((long long)w.n + w.g + w.l)) + 1;
      it.f_hi[1] = min(causal_hi, fdiv(p0 - ((long long)w.n + w.g) - (BK - 1)));
    }
    it.f_lo[2] = 0; it.f_hi[2] = min(causal_hi, w.s >= BK ? (w.s - BK) / BK : -1);
  }
  return it.nt > 0;
}

// How the items are handed out (FORM).
//   kTakenOver  an item per number of the grid; a block takes over the numbers whose blocks have not started
//   kSplit      two blocks, a cluster, share one item (few items, long lists): each takes half of its steps, and the partial
//               states are merged through distributed shared memory
//   kShares     as the first, but the first `starters` numbers stand for `rounds` items each, from alternate ends.  A number
//               taken over costs a block up to a microsecond between two items, more than short lists hide, and so do the
//               numbers past a packed batch's last item (us, a fixed share of all / all taken over / three quarters in
//               shares: 100 prompts of 200 tokens, 16 heads 73 / 78 / 75; 300 of 130, 32 heads 329 / 362 / 316; 48 of 60
//               to 5000 425 / 430 / 407; 64 of 1000, local 128 496 / 573 / 481)
constexpr int kTakenOver = 0, kSplit = 1, kShares = 2;
template <int D, bool VARLEN, int FORM>
__global__ void __launch_bounds__(kPairThreads, 1)
cowa_fwd_pair_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                     const __grid_constant__ CUtensorMap tmV, const __grid_constant__ CUtensorMap tmO,
                     const __grid_constant__ FwdArgs a, const int starters, const int rounds) {
  using SM = PairSmem<D>;
  constexpr bool SPLIT = FORM == kSplit, SHARES = FORM == kShares;
  constexpr int NSLAB = D / 64;        // 64-element (128-byte) slabs along D
  constexpr int SLAB = 128 * 128;      // bytes of one slab of a 128-row tile
  constexpr uint32_t TMEM_COLS = 512;  // S/P of head x: [128x, 128x + 128); O of head x: [256 + 128x, ... + D)
  constexpr uint32_t cO = 256;
  constexpr uint32_t IDESC_S2 = idesc_bf16(128, BS, 0, 0), IDESC_S1 = idesc_bf16(128, BK, 0, 0);
  constexpr uint32_t IDESC_O = idesc_bf16(128, D, 0, 1);

  if constexpr (!SPLIT) grid_wait();
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* sQ = smem + SM::oQ;      // [2 heads][kQ]
  uint8_t* sK = smem + SM::oK;      // [2][kKV]
  uint8_t* sV = smem + SM::oV;      // [2][kKV]
  uint8_t* sOut = smem + SM::oOut;
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + SM::oBar);
  uint64_t* bar_q_full = bars + 0;    //     Q of an item has landed
  uint64_t* bar_q_empty = bars + 1;   //     every S of the item has been computed
  uint64_t* bar_k_full = bars + 2;    // [2]
  uint64_t* bar_k_empty = bars + 4;   // [2]
  uint64_t* bar_v_full = bars + 6;    // [2]
  uint64_t* bar_v_empty = bars + 8;   // [2]
  uint64_t* bar_s = bars + 10;        // [2 heads] S of a step is in TMEM
  uint64_t* bar_p = bars + 12;        // [2 heads][2 halves] count 4 (warps): P written over S
  uint64_t* bar_o_full = bars + 16;   // [2 heads] O of an item is complete
  uint64_t* bar_o_empty = bars + 18;  // [2 heads] count 4: O has been read
  uint64_t* bar_i_full = bars + 20;   // [2] a work item has been published
  uint64_t* bar_i_empty = bars + 22;  // [2] count kItemReaders: it has been read
  uint64_t* bar_next = bars + 24;     //     the next item's number is here
  uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(bars + 25);

  const int tid = threadIdx.x;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);  // warp-uniform by construction

  if (tid == 0) {
    for (int s = 0; s < 25; ++s)
      mbar_init(bars + s, (s >= 12 && s < 16) || s == 18 || s == 19 ? 4 : s == 22 || s == 23 ? kItemReaders : 1);
    fence_mbar_init();
  }
  if (warp == 9 && !SPLIT) {
    __syncwarp();
    tmem_alloc(tmem_holder, TMEM_COLS);
    tmem_relinquish();
  }
  if constexpr (SPLIT) {
    // One short item a block: the TMA warp works out a batched call's item ahead of the wait for the kernel before, and does not
    // wait for TMEM, which is allocated behind it (see cowa_fwd_kernel).  512 tokens behind 32K 54 -> 52.6 us.  (The other forms
    // lose up to a hundredth so, in registers.)
    if (tid == 256) { prefetch_tmap(&tmQ); prefetch_tmap(&tmK); prefetch_tmap(&tmV); }
    __syncthreads();
    if (warp == 8) {
      asm volatile("bar.arrive 3, 384;" ::: "memory");
      if (VARLEN) grid_enter();
    } else {
      grid_enter();
      if (warp == 9) {
        __syncwarp();
        tmem_alloc(tmem_holder, TMEM_COLS);
        tmem_relinquish();
      }
      tc_fence_before();
      asm volatile("bar.sync 3, 384;" ::: "memory");
    }
  } else {
    tc_fence_before();
    __syncthreads();
  }
  tc_fence_after();
  const uint32_t tb = SPLIT && warp == 8 ? 0u : *tmem_holder;

  bool ok = true;  // false once a bounded wait ran out; every role then falls through to the teardown
  auto warp_arrive = [&](uint64_t* bar) {  // one arrival for the whole warp
    __syncwarp();
    if ((tid & 31) == 0) mbar_arrive(bar);
  };
  // Work item number ni of this block; false when a wait ran out or there is none left.  Its words pass through a
  // shuffle so that the compiler knows them to be uniform over the warp (branches and counters on the uniform path).
  auto next_item = [&](uint32_t ni, PairItem& it) -> bool {
    ok = mbar_wait(bar_i_full + (ni & 1), (ni >> 1) & 1, a.status);
    if (!ok) return false;
    const int* src = reinterpret_cast<const int*>(smem + SM::oItem + (ni & 1) * 128);
    int words[sizeof(PairItem) / 4];
#pragma unroll
    for (int i = 0; i < (int)(sizeof(PairItem) / 4); ++i) words[i] = __shfl_sync(0xFFFFFFFFu, src[i], 0);
    __syncwarp();
    if ((tid & 31) == 0) mbar_arrive(bar_i_empty + (ni & 1));
    memcpy(&it, words, sizeof(PairItem));
    return it.nt > 0;
  };

  // Registers: 168 a thread at launch; the softmax threads hold a row of S: 2 * 208 + 88 = 3 * 168.
  if (warp >= 8) {
   setmaxnreg_dec<88>();
   if (warp == 8) {
    // ======================= TMA producer =======================
    const bool lead = elect_one();
    if (!SPLIT && lead) { prefetch_tmap(&tmQ); prefetch_tmap(&tmK); prefetch_tmap(&tmV); }
    int c = 0;       // steps loaded so far, all items together: step c uses slot c & 1
    uint32_t ni = 0;  // items so far
    // The grid has a number per item, heaviest items first (SHARES: fewer).  A block starts with its own and, towards the end
    // of an item, takes over the next one whose block has not started: lists differ in length, and with a fixed share of the
    // items per block the last SM was busy 20 % longer than the average one (one KV head of 20001 tokens), 25 % for packed
    // prompts.
    uint32_t asked = 0, answered = 0;  // requests
    auto ask = [&]() {
      if (lead) {
        mbar_expect_tx(bar_next, 16);
        clc_request(smem + SM::oNext, bar_next);
      }
      ++asked;
    };
    auto next_index = [&]() -> int {
      answered = asked;
      if (!mbar_wait(bar_next, (asked - 1) & 1, a.status)) { ok = false; return -1; }
      const int x = __shfl_sync(0xFFFFFFFFu, clc_block(smem + SM::oNext), 0);
      fence_proxy_async_smem();  // read before the next answer is written
      __syncwarp();
      return x;
    };
    int idx = SPLIT ? blockIdx.x / 2 : blockIdx.x;
    int num = idx, rnd = 0;  // SHARES: this block's number, and how many of its items came before
    int past = 0x7FFFFFFF;   // ... from this item on there are none
    if (SHARES && num >= starters) idx += (rounds - 1) * starters;
    auto more = [&]() { return SHARES && num < starters && rnd + 1 < rounds; };
    auto next_item_index = [&]() -> int {
      if (more()) {
        ++rnd;
        return rnd * starters + ((rnd & 1) ? starters - 1 - num : num);
      }
      const int x = next_index();
      num = x; rnd = 0;
      return SHARES && x >= starters ? x + (rounds - 1) * starters : x;
    };
    while (ok) {
      PairItem& it = *reinterpret_cast<PairItem*>(smem + SM::oItem + (ni & 1) * 128);
      {
        PairItem mine;
        if (SPLIT) {
          if (ni > 0) break;
          if (locate_item<VARLEN>(a, idx, mine)) {
            const int n = (mine.nt + 1) >> 1, rank = (int)cluster_rank();
            mine.t0 = 2 * (n * rank / 2);
            mine.nt = max(min(2 * (n * (rank + 1) / 2), mine.nt) - mine.t0, 0);
          } else {
            mine.nt = mine.work = 0;
          }
        } else if (idx < 0) {
          mine.nt = 0;
        } else if ((SHARES && idx >= past) || !locate_item<VARLEN>(a, idx, mine)) {
          if (SHARES && idx < past && mine.b < 0) past = idx;
          if (!more()) ask();
          idx = next_item_index();
          continue;
        }
        if (SPLIT && !VARLEN) grid_enter();
        if (SHARES && mine.nt > 0 && mine.nt <= 6 && !more()) ask();  // of up to three steps: no later moment is early enough
        if (ni >= 2) ok = mbar_wait(bar_i_empty + (ni & 1), ((ni >> 1) & 1) ^ 1, a.status);
        if (!ok) break;
        if (lead) {
          it = mine;
          mbar_arrive(bar_i_full + (ni & 1));
        }
        __syncwarp();
        if (mine.nt == 0) break;
      }
      auto load_kv = [&](uint8_t* base, const CUtensorMap* tm, uint64_t* bar, int t) {
        if (lead) {
          const int nh = t + 1 < it.nt ? 2 : 1;
          mbar_expect_tx(bar, nh * (SM::kKV / 2));
          for (int hf = 0; hf < nh; ++hf) {
            const int row = it.kbase + cowa_fwd_tile_at(it.rg, it.t0 + t + hf) * BK;
            for (int s = 0; s < NSLAB; ++s) tma_load_4d(base + s * SLAB + hf * (SLAB / 2), tm, bar, s * 64, row, it.hk, it.bt);
          }
        }
      };
      const int ask_at = max((it.nt - 1) / 2 - 2, 0) * 2;  // two steps before the last
      for (int t = 0; t < it.nt; t += 2, ++c) {
        const int sl = c & 1;
        const uint32_t ph = ((c >> 1) & 1) ^ 1;
        if (c >= 2) ok = mbar_wait(bar_k_empty + sl, ph, a.status);
        if (!ok) break;
        // a microsecond or more before the answer is needed
        if (!SPLIT && t == ask_at && (!SHARES || (it.nt > 6 && !more()))) ask();
        load_kv(sK + sl * SM::kKV, &tmK, bar_k_full + sl, t);
        if (t == 0) {
          if (ni > 0) ok = mbar_wait(bar_q_empty, (ni - 1) & 1, a.status);
          if (!ok) break;
          if (lead) {
            mbar_expect_tx(bar_q_full, 2 * SM::kQ);
            for (int x = 0; x < 2; ++x)
              for (int s = 0; s < NSLAB; ++s)
                tma_load_4d(sQ + x * SM::kQ + s * SLAB, &tmQ, bar_q_full, s * 64, it.qbase + it.q0, it.h0 + x, it.bt);
          }
        }
        if (c >= 2) ok = mbar_wait(bar_v_empty + sl, ph, a.status);
        if (!ok) break;
        load_kv(sV + sl * SM::kKV, &tmV, bar_v_full + sl, t);
      }
      ++ni;
      if (!SPLIT && ok) idx = next_item_index();
    }
    if (asked != answered) mbar_wait(bar_next, (asked - 1) & 1, a.status);  // (a wait ran out) no answer may come later
   } else if (warp == 9) {
    // ======================= MMA issuer (warp-uniform control flow, one elected lane issues) =======================
    const bool lead = elect_one();
    const uint64_t dQ0 = smem_desc_sw128(smem_u32(sQ), 16, 1024);    // Q, K-major (A of S)
    const uint64_t dK0 = smem_desc_sw128(smem_u32(sK), 16, 1024);    // K, K-major (B of S)
    const uint64_t dV0 = smem_desc_sw128(smem_u32(sV), SLAB, 1024);  // V, MN-major (B of O)
    constexpr uint32_t kQ16 = SM::kQ >> 4, kKV16 = SM::kKV >> 4;
    int c = 0;
    uint32_t ni = 0;
    PairItem it;
    for (; ok && !(SPLIT && ni > 0) && next_item(ni, it); ++ni) {
      const int nt = it.nt;
      const int n = (nt + 1) >> 1;  // steps
      auto issue_s = [&](int x, int t, int sl) {  // S_x = Q_x K^T of step t; 64 keys only in an odd last step
        if (lead) {
          const uint32_t id = 2 * t + 1 < nt ? IDESC_S2 : IDESC_S1;
          const uint64_t dA = dQ0 + x * kQ16, dB = dK0 + sl * kKV16;
#pragma unroll
          for (int kk = 0; kk < D / 16; ++kk)
            mma_ss(tb + x * 128, dA + (((kk / 4) * SLAB + (kk % 4) * 32) >> 4), dB + (((kk / 4) * SLAB + (kk % 4) * 32) >> 4),
                   id, kk > 0);
          mma_commit(bar_s + x);
          if (x == 1) {
            mma_commit(bar_k_empty + sl);
            if (t == n - 1) mma_commit(bar_q_empty);
          }
        }
      };
      ok = mbar_wait(bar_k_full + (c & 1), (c >> 1) & 1, a.status) && mbar_wait(bar_q_full, ni & 1, a.status);
      if (!ok) break;
      tc_fence_after();
      issue_s(0, 0, c & 1);
      issue_s(1, 0, c & 1);
      for (int t = 0; t < n && ok; ++t, ++c) {
        const int sl = c & 1;
        const uint32_t par = (c >> 1) & 1, sp = c & 1;  // slot parity; parity of this step's S and P
        const bool two = 2 * t + 1 < nt;
        ok = mbar_wait(bar_v_full + sl, par, a.status);
        if (!ok) break;
#pragma unroll
        for (int x = 0; x < 2; ++x) {
          if (t == 0 && ni > 0) {
            ok = mbar_wait(bar_o_empty + x, (ni - 1) & 1, a.status);
            if (!ok) break;
          }
          ok = mbar_wait(bar_p + 2 * x, sp, a.status);
          if (!ok) break;
          tc_fence_after();
          const uint64_t dB = dV0 + sl * kKV16;
          if (lead) {
#pragma unroll
            for (int kk = 0; kk < 2 * kSplitQ + 2; ++kk)
                mma_ts(tb + cO + x * 128, tb + x * 128 + kk * 8, dB + ((kk * 2048) >> 4), IDESC_O, (t > 0 || kk > 0) ? 1u : 0u);
          }
          ok = mbar_wait(bar_p + 2 * x + 1, sp, a.status);
          if (!ok) break;
          tc_fence_after();
          if (lead) {
            if (two) {
#pragma unroll
              for (int kk = 2 * kSplitQ + 2; kk < 8; ++kk)
                mma_ts(tb + cO + x * 128, tb + x * 128 + kk * 8, dB + ((kk * 2048) >> 4), IDESC_O, 1u);
            }
            if (t == n - 1) mma_commit(bar_o_full + x);
            if (x == 1) mma_commit(bar_v_empty + sl);
          }
          if (t + 1 < n) {
            if (x == 0) {
              ok = mbar_wait(bar_k_full + (sl ^ 1), ((c + 1) >> 1) & 1, a.status);
              if (!ok) break;
              tc_fence_after();
            }
            issue_s(x, t + 1, sl ^ 1);
          }
        }
      }
    }
   }
   if constexpr (SPLIT) {  // the softmax warps' merge
     cluster_sync();
     cluster_sync();
   }
  } else {
    setmaxnreg_inc<208>();
    // ======================= softmax: one query row per thread =======================
    const int x = warp >> 2;                                              // head of the pair
    const int r = tid & 127;                                              // row of the tile = TMEM lane
    const uint32_t t_lane = tb + ((uint32_t)((warp & 3) * 32) << 16);
    const uint32_t t_S = t_lane + x * 128, t_O = t_lane + cO + x * 128;
    const float2 sc2 = make_float2(a.scale_log2, a.scale_log2);
    uint8_t* stage = sOut + x * SM::kOut;
    bool stored = false;  // (first thread) a bulk store from `stage` may still be reading it
    int c = 0;
    uint32_t ni = 0;
    PairItem it;
    for (; ok && !(SPLIT && ni > 0) && next_item(ni, it); ++ni) {
      const int n = (it.nt + 1) >> 1, q0 = it.q0, off = it.off, Nk = it.Nk;
      const int row = q0 + r;
      const bool row_valid = row < it.Nq;
      const int rowpos = row + off;  // position of this query on the key axis
      float m_ref = -INFINITY, l_sum = 0.f;

      // The two tiles of step t (the second one only if `two`), and whether both need no mask; straight-line code, so
      // that it overlaps with the exponentials of the step before.
      const int n0 = cowa_range_len(it.rg[0]), n1 = n0 + cowa_range_len(it.rg[1]);
      struct Step { int ja, jb; bool two, full; } cur;
      auto step_at = [&](int t) {
        auto at = [&](int u, bool* full) {
          const int j = u < n0 ? it.rg[0].hi - u : u < n1 ? it.rg[1].hi + n0 - u : it.rg[2].hi + n1 - u;
          const int lo = u < n0 ? it.f_lo[0] : u < n1 ? it.f_lo[1] : it.f_lo[2];
          const int hi = u < n0 ? it.f_hi[0] : u < n1 ? it.f_hi[1] : it.f_hi[2];
          *full = j >= lo && j <= hi;
          return j;
        };
        Step st;
        bool fa, fb;
        st.ja = at(it.t0 + 2 * t, &fa);
        st.jb = at(it.t0 + 2 * t + 1, &fb);
        st.two = 2 * t + 1 < it.nt;
        st.full = fa && fb && st.two;
        return st;
      };
      Step nxt = step_at(0);

      for (int t = 0; t < n && ok; ++t, ++c) {
        cur = nxt;
        const int ja = cur.ja, jb = cur.jb;
        const bool two = cur.two;
        ok = mbar_wait(bar_s + x, c & 1, a.status);
        if (!ok) break;
        tc_fence_after();
        uint32_t sr[4][32];
#pragma unroll
        for (int q = 0; q < 4; ++q) tmem_ld32(t_S + q * 32, sr[q]);
        tmem_wait_ld();

        // Boundary steps: each warp looks at its 32 rows x 32 keys; most such squares are all legal.
        if (__builtin_expect(!cur.full, 0)) {
          const CowaWin w = it.w;
          const int kend = row_valid ? min(rowpos, Nk - 1) : -1;  // last causal key of this row
          const int near_lo = rowpos - w.n + 1, sink_hi = min(w.s - 1, kend);
          const int long_hi = w.l > 0 ? min(rowpos - (w.n + w.g), kend) : -1, long_lo = rowpos - (w.n + w.g + w.l) + 1;
          uint32_t mk[4];
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const int base = (q < 2 ? ja : jb) * BK + (q & 1) * 32;
            mk[q] = interval_bits(near_lo, kend, base) | interval_bits(0, sink_hi, base) | interval_bits(long_lo, long_hi, base);
            if (q >= 2 && !two) mk[q] = 0u;
          }
#pragma unroll
          for (int q = 0; q < 4; ++q)
            if (__any_sync(0xFFFFFFFFu, mk[q] != 0xFFFFFFFFu)) {
#pragma unroll
              for (int e = 0; e < 32; ++e)
                if (!((mk[q] >> e) & 1u)) sr[q][e] = 0xFF800000u;  // -inf
            }
        }
        float mxa[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
          for (int e = 0; e < 32; e += 2)
            mxa[(e >> 1) & 3] = max3(mxa[(e >> 1) & 3], __uint_as_float(sr[q][e]), __uint_as_float(sr[q][e + 1]));
        const float mx = fmaxf(fmaxf(mxa[0], mxa[1]), fmaxf(mxa[2], mxa[3])) * a.scale_log2;
        // The reference moves rarely: the row sum, and the accumulator of a warp with such a row, are rescaled then.
        const bool moved = mx > m_ref + 8.f;
        if (__builtin_expect(__any_sync(0xFFFFFFFFu, moved), 0)) {
          const float alpha = moved ? ex2(m_ref - mx) : 1.f;
          if (moved) m_ref = mx;
          l_sum *= alpha;
          const float2 al2 = make_float2(alpha, alpha);
#pragma unroll 1
          for (int q = 0; q < (t > 0 ? D / 16 : 0); ++q) {
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

        if constexpr (VARLEN) {
          // rows after the sequence's last key belong to the next sequence: P is exactly zero there, but
          // 0 x (Inf or NaN) would poison this one, so those V rows are cleared before the product may start
          // (both heads' warps write the same zeros; the slot is released only after both heads' products)
#pragma unroll
          for (int hf = 0; hf < 2; ++hf) {
            const int vrows = Nk - (hf ? jb : ja) * BK;
            if (vrows < BK && (hf == 0 || two)) {
              ok = mbar_wait(bar_v_full + (c & 1), (c >> 1) & 1, a.status);
              if (!ok) break;
              uint8_t* vt = sV + (c & 1) * SM::kKV + hf * (SLAB / 2);
              const int nchunk = (BK - vrows) * 8;  // 16-byte chunks per slab
              for (int s_ = 0; s_ < NSLAB; ++s_)
                for (int c_ = r; c_ < nchunk; c_ += 128)
                  *reinterpret_cast<uint4*>(vt + s_ * SLAB + vrows * 128 + c_ * 16) = make_uint4(0u, 0u, 0u, 0u);
              fence_proxy_async_smem();
            }
          }
          if (!ok) break;
        }

        // p = 2^(s * scale - m): packed fp32 pairs for the multiply-add and the row sum
        const float sub = (m_ref == -INFINITY) ? 0.f : m_ref;
        const float2 nsub2 = make_float2(-sub, -sub);
        float2 rsa[4] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
        nxt = step_at(t + 1);
        // The exponentials of a 32-key group are issued between the sums and conversions of the group before it, so
        // that the special-function unit does not wait for them.
#pragma unroll
        for (int q = 0; q < 5; ++q) {
          uint32_t pk[16];
#pragma unroll
          for (int e = 0; e < 32; e += 2) {
            if (q < 4) {
              const float2 y = fma2(make_float2(__uint_as_float(sr[q & 3][e]), __uint_as_float(sr[q & 3][e + 1])), sc2, nsub2);
              const float2 z = e % 16 == 0 ? exp2_fma(y) : make_float2(ex2(y.x), ex2(y.y));
              sr[q & 3][e] = __float_as_uint(z.x);
              sr[q & 3][e + 1] = __float_as_uint(z.y);
            }
            if (q > 0) {
              const float2 pp = make_float2(__uint_as_float(sr[(q - 1) & 3][e]), __uint_as_float(sr[(q - 1) & 3][e + 1]));
              rsa[(e >> 1) & 3] = add2(rsa[(e >> 1) & 3], pp);
              pk[e / 2] = pack_bf16(pp.x, pp.y);
            }
          }
          if (q > 0) tmem_st16(t_S + (q - 1) * 16, pk);
          if (q - 1 == kSplitQ) {  // the first half of P is in place
            tmem_wait_st();
            tc_fence_before();
            warp_arrive(bar_p + 2 * x);
          }
        }
        const float2 rs2 = add2(add2(rsa[0], rsa[1]), add2(rsa[2], rsa[3]));
        l_sum += rs2.x + rs2.y;
        tmem_wait_st();
        tc_fence_before();
        warp_arrive(bar_p + 2 * x + 1);
      }
      if (!ok) break;

      // ---- epilogue: O / l, LSE ----
      ok = mbar_wait(bar_o_full + x, ni & 1, a.status);
      if (!ok) break;
      if constexpr (SPLIT) {
        // fp32 O goes where K and V were, once both heads' products have read them; the row's state where Q was
        ok = mbar_wait(bar_o_full + (x ^ 1), ni & 1, a.status);
        if (!ok) break;
        tc_fence_after();
        uint8_t* orow = sK + (x * BQ + r) * (D * 4);
#pragma unroll
        for (int q = 0; q < D / 32; ++q) {
          uint32_t ov[32];
          tmem_ld32(t_O + q * 32, ov);
          tmem_wait_ld();
#pragma unroll
          for (int e = 0; e < 8; ++e)
            *reinterpret_cast<uint4*>(orow + (((q * 8 + e) ^ (r & 7)) << 4)) =
                make_uint4(ov[e * 4], ov[e * 4 + 1], ov[e * 4 + 2], ov[e * 4 + 3]);
        }
        reinterpret_cast<float2*>(sQ)[x * BQ + r] = make_float2(m_ref, l_sum);
        continue;
      }
      tc_fence_after();
      const float inv = l_sum > 0.f ? 1.f / l_sum : 0.f;
      uint32_t ob[D / 2];
#pragma unroll
      for (int q = 0; q < D / 32; ++q) {
        uint32_t ov[32];
        tmem_ld32(t_O + q * 32, ov);
        tmem_wait_ld();
#pragma unroll
        for (int e = 0; e < 32; e += 2)
          ob[q * 16 + e / 2] = pack_bf16(__uint_as_float(ov[e]) * inv, __uint_as_float(ov[e + 1]) * inv);
      }
      tc_fence_before();
      warp_arrive(bar_o_empty + x);
      const int h = it.h0 + x;
      if (row_valid) {
        const size_t li = VARLEN ? (size_t)h * a.total_q + it.qbase + row : ((size_t)it.b * a.Hq + h) * it.Nq + row;
        a.lse[li] = 0.6931471805599453f * (m_ref + log2f(l_sum));
      }
      if (VARLEN && q0 + BQ > it.Nq) {  // written row by row: the rows after the sequence's last belong to another one
        if (row_valid) {
          uint4* dst = reinterpret_cast<uint4*>(a.o + ((size_t)h * a.total_q + it.qbase + row) * D);
#pragma unroll
          for (int q = 0; q < D / 8; ++q) dst[q] = make_uint4(ob[q * 4], ob[q * 4 + 1], ob[q * 4 + 2], ob[q * 4 + 3]);
        }
      } else {
#pragma unroll
        for (int s = 0; s < NSLAB; ++s) {
          if (r == 0 && stored) tma_wait_group_read<0>();
          asm volatile("bar.sync %0, 128;" ::"r"(1 + x) : "memory");
#pragma unroll
          for (int q = 0; q < 8; ++q)
            *reinterpret_cast<uint4*>(stage + r * 128 + ((q ^ (r & 7)) << 4)) =
                make_uint4(ob[s * 32 + q * 4], ob[s * 32 + q * 4 + 1], ob[s * 32 + q * 4 + 2], ob[s * 32 + q * 4 + 3]);
          fence_proxy_async_smem();
          asm volatile("bar.sync %0, 128;" ::"r"(1 + x) : "memory");
          if (r == 0) {
            tma_store_4d(&tmO, stage, s * 64, it.qbase + q0, h, it.bt);
            tma_commit_group();
            stored = true;
          }
        }
      }
    }
    if (r == 0 && stored) tma_wait_group_read<0>();

    if constexpr (SPLIT) {
      // Merge of the two blocks' partial states: block `rank` writes head `rank`, a warp 16 rows, all of the other block's O of them in
      // flight together.  (A row at a time and lane, 32 rows an access: 2 us longer.  Four rows of one block after the other,
      // the block's own through the cluster's window, too: 61.0 instead of 59.3 us for 512 tokens behind 32K.)
      const PairItem& item = *reinterpret_cast<const PairItem*>(smem + SM::oItem);
      const int rank = (int)cluster_rank(), lane = tid & 31;
      if (item.nt == 0) reinterpret_cast<float2*>(sQ)[tid] = make_float2(-INFINITY, 0.f);
      cluster_sync();
      if (item.work > 0) {
        const int r0 = rank * BQ + warp * 16;  // of the 2 x 128
        const int steps = (item.work + 1) >> 1, here = rank == 0 ? steps / 2 : steps - steps / 2;
        const uint32_t other = map_cluster(smem_u32(sK) + r0 * (D * 4), rank ^ 1);
        const uint8_t* const own = sK + r0 * (D * 4);
        float4 v[16];
#pragma unroll
        for (int u = 0; u < 16; ++u)  // (a block without a step left no O)
          v[u] = here < steps ? ld_cluster_f4(other + u * (D * 4) + ((lane ^ (u & 7)) << 4)) : make_float4(0.f, 0.f, 0.f, 0.f);
        const float2 mine = reinterpret_cast<const float2*>(sQ)[r0 + (lane & 15)];
        const float2 theirs = ld_cluster_f2(map_cluster(smem_u32(sQ) + (r0 + (lane & 15)) * 8, rank ^ 1));
        const float M = fmaxf(mine.x, theirs.x);
        float wa = mine.x == -INFINITY ? 0.f : ex2(mine.x - M), wb = theirs.x == -INFINITY ? 0.f : ex2(theirs.x - M);
        const float L = fmaf(theirs.y, wb, mine.y * wa), inv = L == 0.f ? 0.f : 1.f / L;  // a NaN sum has to come out as NaN
        wa *= inv; wb *= inv;
        const int row0 = item.q0 + warp * 16, h = item.h0 + rank;
        if (lane < 16 && row0 + lane < item.Nq) {
          const size_t li = VARLEN ? (size_t)h * a.total_q + item.qbase + row0 + lane : ((size_t)item.b * a.Hq + h) * item.Nq + row0 + lane;
          a.lse[li] = 0.6931471805599453f * (M + log2f(L));
        }
        __nv_bfloat16* const dst = a.o + (VARLEN ? ((size_t)h * a.total_q + item.qbase + row0) * D
                                                 : (size_t)item.b * a.so.b + (size_t)h * a.so.h + (size_t)row0 * a.so.t) + lane * 4;
        const long long step = VARLEN ? D : a.so.t;
#pragma unroll
        for (int u = 0; u < 16; ++u) {
          const float4 x = here > 0 ? *reinterpret_cast<const float4*>(own + u * (D * 4) + ((lane ^ (u & 7)) << 4)) : make_float4(0.f, 0.f, 0.f, 0.f);
          const float w0 = __shfl_sync(0xFFFFFFFFu, wa, u), w1 = __shfl_sync(0xFFFFFFFFu, wb, u);
          if (row0 + u < item.Nq)
            *reinterpret_cast<uint2*>(dst + u * step) = make_uint2(pack_bf16(fmaf(v[u].x, w1, x.x * w0), fmaf(v[u].y, w1, x.y * w0)),
                                                                   pack_bf16(fmaf(v[u].z, w1, x.z * w0), fmaf(v[u].w, w1, x.w * w0)));
        }
      }
      cluster_sync();  // no block leaves while another one reads its shared memory
    }
  }

  // ---- teardown ----
  tc_fence_before();
  __syncthreads();
  if (warp == 9) {
    __syncwarp();
    tmem_dealloc(tb, TMEM_COLS);
  }
}

}  // namespace

namespace cowa {

int resident_pairs() {
  static std::atomic<int> cache[64];  // per device
  int dev = 0, n = 0;
  if (cudaGetDevice(&dev) == cudaSuccess && dev >= 0 && dev < 64) {
    n = cache[dev].load(std::memory_order_relaxed);
    if (n > 0) return n;
    const auto kernel = cowa_fwd_pair_kernel<128, false, kSplit>;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(2); cfg.blockDim = dim3(kPairThreads); cfg.dynamicSmemBytes = PairSmem<128>::kBytes;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr; cfg.numAttrs = 1;
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, PairSmem<128>::kBytes) == cudaSuccess &&
        cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) == cudaSuccess && n > 0) {
      cache[dev].store(n, std::memory_order_relaxed);
      return n;
    }
  }
  cudaGetLastError();
  return 72;
}

template <int D, bool VARLEN>
int launch_fwd_pair(const CUtensorMap& mq, const CUtensorMap& mk, const CUtensorMap& mv, const CUtensorMap& mo,
                    const FwdArgs& a, long long items, int rounds, int split, cudaStream_t st) {
  auto kernel = cowa_fwd_pair_kernel<D, VARLEN, kSplit>;
  if constexpr (D == 128) {
    if (split == 1) kernel = cowa_fwd_pair_kernel<D, VARLEN, kTakenOver>;
    if constexpr (VARLEN) {
      if (split == 1 && rounds > 1) kernel = cowa_fwd_pair_kernel<D, VARLEN, kShares>;
    }
  }
  COWA_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, PairSmem<D>::kBytes));
  cudaLaunchConfig_t cfg = {};
  const int starters = (int)std::min<long long>(items, sm_count());
  cfg.gridDim = dim3((unsigned)(split > 1 ? items * split : items - (rounds - 1ll) * starters));
  cfg.blockDim = dim3(kPairThreads); cfg.dynamicSmemBytes = PairSmem<D>::kBytes; cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = (unsigned)split; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr; cfg.numAttrs = split > 1 ? 2 : 1;
  COWA_CUDA_TRY(cudaLaunchKernelEx(&cfg, kernel, mq, mk, mv, mo, a, starters, rounds));
  return COWA_OK;
}

#define COWA_INSTANTIATE(D, V)                                                                                          \
  template int launch_fwd_pair<D, V>(const CUtensorMap&, const CUtensorMap&, const CUtensorMap&, const CUtensorMap&,    \
                                     const FwdArgs&, long long, int, int, cudaStream_t);
COWA_INSTANTIATE(128, false)
COWA_INSTANTIATE(128, true)
#undef COWA_INSTANTIATE

}  // namespace cowa
