// CoWindow Attention forward (Algorithm 1) for sm_100a.
//
// One thread block = one (batch, QO head, 128-row QO tile); it walks the tile's visited KV tiles
// J_h(i) (analytic scheduler, descending order) in steps of 64 keys.  Five warps:
//   warps 0-3  softmax: one query row per thread.  tcgen05.ld of S, (boundary tiles only) the
//              window/causal mask from a per-row bit mask, online softmax in base 2 with the
//              scale folded in, P written back to TMEM as bf16 over S's columns.
//   warp 4     control (one lane): TMA loads of K and V (128B swizzle, two buffers each) and all
//              tcgen05.mma issue: S = Q K^T into one of two TMEM buffers, O += P V with P as the
//              TMEM operand.  S of step t+1 is issued before the softmax of step t starts, so the
//              softmax threads never wait for the tensor pipe in steady state.
// The running max is only advanced when the row max grows by more than 2^8 (the accumulator is
// rescaled in TMEM only then); the final normalisation uses the same reference max, so the
// result is the exact softmax.  The QO heads of a GQA group at the same tile are adjacent in launch
// order and share K/V through L2.
// At D = 128 two such blocks fit an SM (96 KB shared memory, 256 TMEM columns each).  At D = 64 the exponentials bound the
// kernel and the chain of one step (1600 clocks: S landed 320, load and row maximum 210, exponentials 720 where the
// special-function unit needs 512, hand-over 280) leaves the unit idle: with one S buffer a block takes 128 columns and
// 50 KB, four are resident, and S(t+1) is issued behind O += P V of step t.  An SM then takes a step in 490 clocks (two blocks
// with two buffers: 800 at the same clock rate); us, before / now: 640 blocks of up to 40 steps 50.9 / 42.6, 1920 of 35
// 126 / 107, 8896 of 90 (power-limited, 1.3 GHz) 1365 / 1265.
// Where blocks are too few to fill the chip (see the rule in launch_fwd), the last two cutting a list into parts:
//   NB = 2   two S buffers and two blocks per SM, where two or three are all an SM gets (D = 64);
//   NS = 4   four streams, each the five warps above with slots and TMEM of its own, in one block (D = 64);
//   SPLIT    a cluster of 2, 4 or 8 blocks, each with two S buffers, as latency counts and not the number of blocks.
// A part keeps its own reference and accumulator; they are merged through (distributed) shared memory.
// The same kernel serves N_q <= N_k (queries bottom-right aligned) and, with VARLEN, packed batches
// [H, total, D] whose sequences have their own N_q <= N_k: a block then finds its (sequence, tile) by a
// warp scan of the offset arrays and stores a sequence's last, partial tile row by row.
#include <cuda_bf16.h>

#include "cowa_fwd.h"

#include <algorithm>
#include <type_traits>

using namespace cowa_ptx;

namespace {

constexpr int BQ = 128, BK = 64;
constexpr int kFwdThreads = 160;

template <int D, int NS, bool SPLIT>
struct FwdSmem {
  static constexpr int kQ = BQ * D * 2;   // Q tile (later the O staging tile)
  static constexpr int kKV = BK * D * 2;  // one K or V step tile
  static constexpr int oQ = 0, oKV = kQ, oState = kQ + NS * 4 * kKV, oBar = oState + (NS > 1 || SPLIT ? NS * BQ * 8 : 0);
  static constexpr int kUsed = oBar + 32 + NS * 80 + 1024;  // + barriers + alignment slack
  // A cluster's blocks hold their TMEM, half of an SM's each, until all of them are through, and neither the allocation nor the
  // cluster's barrier is a bounded wait.  A third block on an SM would wait for TMEM that two other clusters hold; if their other
  // blocks waited on other SMs for this cluster's, none would ever end.  So a block takes more than a third of an SM's shared memory
  // whatever its registers allow (50 KB and 131 registers at D = 64: at 128 three would fit).
  static constexpr int kSm = 228 * 1024, kReserved = 1024;  // shared memory of an SM, and what each block takes besides its own
  static constexpr int kBytes = SPLIT ? std::max(kUsed, kSm / 3) : kUsed;
  static_assert(!SPLIT || (3 * (kBytes + kReserved) > kSm && 2 * (kBytes + kReserved) <= kSm), "two blocks of clusters on an SM");
};

// NB: S/P buffers of a stream (64 columns each, then O of D); an SM holds 4 / NB streams.
template <int D, bool VARLEN, int NB, int NS, bool SPLIT>
__global__ void __launch_bounds__(kFwdThreads * NS, 4 / NB / NS)
cowa_fwd_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                const __grid_constant__ CUtensorMap tmV, const __grid_constant__ CUtensorMap tmO,
                const __grid_constant__ FwdArgs a) {
  using SM = FwdSmem<D, NS, SPLIT>;
  constexpr bool MERGE = NS > 1 || SPLIT;
  constexpr int NSLAB = D / 64;          // 64-element (128-byte) slabs along D
  constexpr int SLAB_Q = BQ * 128;       // bytes of one slab of a 128-row tile
  constexpr int SLAB_K = BK * 128;       // ... of a 64-row tile
  constexpr uint32_t cO = 64 * NB, STREAM_COLS = 128 * NB, TMEM_COLS = STREAM_COLS * NS;
  constexpr uint32_t IDESC_S = idesc_bf16(128, BK, 0, 0);
  constexpr uint32_t IDESC_O = idesc_bf16(128, D, 0, 1);

  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* sQ = smem + SM::oQ;
  const int tid = threadIdx.x;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);  // warp-uniform by construction
  const bool control = warp >= 4 * NS;
  const int stream = NS == 1 ? 0 : control ? warp - 4 * NS : warp >> 2;
  uint8_t* sK = smem + SM::oKV + stream * 4 * SM::kKV;  // [2][kKV]
  uint8_t* sV = sK + 2 * SM::kKV;                       // [2][kKV]
  uint64_t* bar_q = reinterpret_cast<uint64_t*>(smem + SM::oBar);
  uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(bar_q + 1);
  uint64_t* bars = bar_q + 4 + stream * 10;
  uint64_t* bar_k = bars + 0;   // [2] K step tile landed
  uint64_t* bar_v = bars + 2;   // [2] V step tile landed
  uint64_t* bar_s = bars + 4;   // [2] S of a step is in TMEM buffer b
  uint64_t* bar_p = bars + 6;   // [2] count 128: P written over S
  uint64_t* bar_pv = bars + 8;  //     O += P V of a step (one S buffer: of the last one) has completed

  // ---- work item (heaviest QO tiles first; the group's heads adjacent) ----
  const int csize = SPLIT ? (int)cluster_size() : 1, rank = SPLIT ? (int)cluster_rank() : 0;
  int idx = blockIdx.x / csize;
  const int g = idx % a.G; idx /= a.G;
  const int hk = idx % a.Hkv; idx /= a.Hkv;
  const int h = hk * a.G + g;
  int b = 0, i = 0;
  if constexpr (!VARLEN) {
    b = idx % a.B; idx /= a.B;
    i = (a.Nq + BQ - 1) / BQ - 1 - idx;
  }
  CowaWin w = a.wins.w[hk];

  // What needs nothing of the kernel before this one is done ahead of the wait for it.  Not so the TMEM allocation: a kernel of
  // another library that lets this one in before it has allocated its own columns would then wait for this one's.
  if (tid == 0) {
    mbar_init(bar_q, 1);
    for (int x = 0; x < NS; ++x)
      for (int s = 0; s < 9; ++s) mbar_init(bar_q + 4 + x * 10 + s, s == 6 || s == 7 ? 128 : 1);
    fence_mbar_init();
  }
  if (control && stream == 0 && elect_one()) { prefetch_tmap(&tmQ); prefetch_tmap(&tmK); prefetch_tmap(&tmV); }
  __syncthreads();
  grid_enter();

  // Sequence geometry.  Packed batches: every sequence has its own N_q <= N_k, its rows start at
  // cu_q[b] / cu_k[b] of a [H, total, D] tensor, and its windows follow from its own N_k.
  int Nq = a.Nq, Nk = a.Nk, qbase = 0, kbase = 0;
  int bt = b;  // batch coordinate of the tensor maps (packed tensors have none)
  bool found = true;
  if constexpr (VARLEN) {
    // idx counts the QO tiles of the packed batch, each sequence's heaviest (last) tile first.
    // Every warp finds its (sequence, tile) by a cooperative scan of the offsets.  The grid is an upper bound.
    int lt = 0, nts = 0, pb;
    found = a.longest_first ? varlen_locate_longest(a.cu_q, a.cu_k, a.B, idx, BQ, 1, 0, &b, &lt, &nts)
                            : varlen_locate(a.cu_q, a.B, idx, BQ, 0, &b, &lt, &nts, &pb);
    if (found) {
      i = nts - 1 - lt;
      qbase = a.cu_q[b]; Nq = a.cu_q[b + 1] - qbase;
      kbase = a.cu_k[b]; Nk = a.cu_k[b + 1] - kbase;
      bt = 0;
      if (Nq > Nk || qbase < 0 || kbase < 0 || qbase + Nq > a.total_q || kbase + Nk > a.total_k) {
        // malformed offsets: report, touch nothing
        if (tid == 0) atomicOr(a.status, (unsigned)COWA_DEV_BAD_SEQLENS);
        found = false;
      }
    }
    if (!found) return;  // (every block of a cluster)
    if (a.full_attn) { w.s = 0; w.n = Nk; w.g = 0; w.l = 0; }
    else if (!a.explicit_windows) w = cowa_default_window(Nk, a.hkv_global, a.hkv_offset + hk, a.sink, a.local);
  }
  const int off = Nk - Nq;
  const int q0 = i * BQ, q1 = min(q0 + BQ, Nq) - 1;
  CowaRange rg[3];
  cowa_fwd_ranges(w, q0, q1, off, Nk, BK, rg);
  const int work = cowa_range_len(rg[0]) + cowa_range_len(rg[1]) + cowa_range_len(rg[2]);
  const int parts = csize * NS, part = rank * NS + stream;
  const int t0 = work * part / parts, nt = work * (part + 1) / parts - t0;  // this part's steps: t0 .. t0 + nt - 1 of the list

  // K or V of step t into its slot (one thread)
  auto load_tile = [&](const CUtensorMap* tm, uint8_t* base, uint64_t* bar, int t) {
    const int j = cowa_fwd_tile_at(rg, t0 + t);
    mbar_expect_tx(bar + (t & 1), SM::kKV);
    for (int s = 0; s < NSLAB; ++s)
      tma_load_4d(base + (t & 1) * SM::kKV + s * SLAB_K, tm, bar + (t & 1), s * 64, kbase + j * BK, hk, bt);
  };
  if (control && elect_one()) {  // the first loads are under way while TMEM is being allocated
    if (stream == 0 && work * ((rank + 1) * NS) / parts > work * (rank * NS) / parts) {  // some stream of the block has a step
      mbar_expect_tx(bar_q, SM::kQ);
      for (int s = 0; s < NSLAB; ++s) tma_load_4d(sQ + s * SLAB_Q, &tmQ, bar_q, s * 64, qbase + q0, h, bt);
    }
    if (nt > 0) { load_tile(&tmK, sK, bar_k, 0); load_tile(&tmV, sV, bar_v, 0); }
    if (nt > 1) load_tile(&tmK, sK, bar_k, 1);
  }
  if (warp == 0) {
    __syncwarp();
    tmem_alloc(tmem_holder, TMEM_COLS);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_holder + stream * STREAM_COLS;

  bool ok = true;  // false once a bounded wait ran out; every role then falls through to the teardown

  if (control) {
    // ======================= control: TMA loads and MMA issue =======================
    // The whole warp runs the loop (uniform control flow keeps descriptors and counters in uniform
    // registers); only the elected lane executes the TMA and tcgen05 instructions.
    if (nt > 0) {
      const bool lead = elect_one();
      const uint32_t tb = tmem_base;
      const uint64_t dQ = smem_desc_sw128(smem_u32(sQ), 16, 1024);                 // Q, K-major (A of S)
      const uint64_t dK0 = smem_desc_sw128(smem_u32(sK), 16, 1024);                // K buffer 0, K-major (B of S)
      const uint64_t dV0 = smem_desc_sw128(smem_u32(sV), SLAB_K, 1024);            // V buffer 0, MN-major (B of O)
      constexpr uint32_t kKV16 = SM::kKV >> 4;
      auto load_k = [&](int t) {
        if (lead) load_tile(&tmK, sK, bar_k, t);
      };
      auto load_v = [&](int t) {
        if (lead) load_tile(&tmV, sV, bar_v, t);
      };
      auto issue_s = [&](int buf) {  // S = Q K^T into TMEM buffer buf from K buffer buf
        if (lead) {
          const uint64_t dK = dK0 + buf * kKV16;
#pragma unroll
          for (int kk = 0; kk < D / 16; ++kk)
            mma_ss(tb + (NB == 2 ? buf * 64 : 0), dQ + (((kk / 4) * SLAB_Q + (kk % 4) * 32) >> 4),
                   dK + (((kk / 4) * SLAB_K + (kk % 4) * 32) >> 4), IDESC_S, kk > 0);
          mma_commit(bar_s + (NB == 2 ? buf : 0));
        }
      };
      ok = mbar_wait(bar_q, 0, a.status) && mbar_wait(bar_k, 0, a.status);
      if (ok) { tc_fence_after(); issue_s(0); }
      if constexpr (NB == 1) {
        // S(t + 1) takes the columns of P(t) and is issued right behind the product that reads it; that S(t) has completed
        // means that the product before it has, too.
        if (nt > 1) load_v(1);
        for (int t = 0; t < nt && ok; ++t) {
          const int b_ = t & 1;
          const uint32_t par = (t >> 1) & 1;
          ok = mbar_wait(bar_s, t & 1, a.status);
          if (!ok) break;
          if (t > 0 && t + 1 < nt) load_v(t + 1);
          if (t + 2 < nt) load_k(t + 2);
          if (t + 1 < nt) ok = mbar_wait(bar_k + (b_ ^ 1), ((t + 1) >> 1) & 1, a.status);
          ok = ok && mbar_wait(bar_v + b_, par, a.status) && mbar_wait(bar_p, t & 1, a.status);
          if (!ok) break;
          tc_fence_after();
          if (lead) {
            const uint64_t dV = dV0 + b_ * kKV16;
#pragma unroll
            for (int kk = 0; kk < BK / 16; ++kk)
              mma_ts(tb + cO, tb + kk * 8, dV + ((kk * 2048) >> 4), IDESC_O, (t > 0 || kk > 0) ? 1u : 0u);
            if (t + 1 == nt) mma_commit(bar_pv);
          }
          if (t + 1 < nt) issue_s(b_ ^ 1);
        }
      } else {
      uint32_t par = 0;  // (t >> 1) & 1
      for (int t = 0; t < nt && ok; ++t) {
        const int b_ = t & 1;
        if (t + 1 < nt) {  // S(t+1): its buffer last held P(t-1), whose product was issued before this one
          ok = mbar_wait(bar_k + (b_ ^ 1), b_ ? (par ^ 1) : par, a.status);
          if (!ok) break;
          tc_fence_after();
          issue_s(b_ ^ 1);
        }
        if (t + 2 < nt) {  // K(t+2) over K(t), once S(t) has been computed
          ok = mbar_wait(bar_s + b_, par, a.status);
          if (!ok) break;
          load_k(t + 2);
        }
        if (t + 1 < nt) {  // V(t+1) over V(t-1), once O += P V of step t-1 has completed
          if (t >= 1) ok = mbar_wait(bar_pv, (t - 1) & 1, a.status);
          if (!ok) break;
          load_v(t + 1);
        }
        ok = mbar_wait(bar_p + b_, par, a.status) && mbar_wait(bar_v + b_, par, a.status);
        if (!ok) break;
        tc_fence_after();
        if (lead) {
          const uint64_t dV = dV0 + b_ * kKV16;
#pragma unroll
          for (int kk = 0; kk < BK / 16; ++kk)
            mma_ts(tb + cO, tb + b_ * 64 + kk * 8, dV + ((kk * 2048) >> 4), IDESC_O, (t > 0 || kk > 0) ? 1u : 0u);
          mma_commit(bar_pv);
        }
        if (b_) par ^= 1;
      }
      }
    }
  } else {
    // ======================= softmax: one query row per thread =======================
    const int r = tid & (BQ - 1);
    const uint32_t t_lane = tmem_base + ((uint32_t)((warp & 3) * 32) << 16);  // this warp's 32 lanes
    const uint32_t t_O = t_lane + cO;
    const int row = q0 + r;
    const bool row_valid = row < Nq;
    // Last, partial tile of a packed sequence: the rows after it belong to the next sequence, so the
    // tile is written row by row instead of by one bulk store.
    const bool tail_rows = VARLEN && (q0 + BQ > Nq);
    const int rowpos = row + off;  // position of this query on the key axis
    float m_ref = -INFINITY, l_sum = 0.f;
    const float2 sc2 = make_float2(a.scale_log2, a.scale_log2);

    // Which visited tiles need no mask?  Inside each of the three ranges these form one interval of tile
    // indices, found once here; the loop then only compares.  The intervals are conservative (a tile that
    // straddles two windows, or sink and non-sink columns, is treated as a boundary tile and masked, which
    // is always correct).  With d = (row position) - (key index): every pair of tile j is causal iff
    // 64 j + 63 <= q0 + off; it lies in the near window iff q1 + off - 64 j < n; in the long window iff also
    // q0 + off - (64 j + 63) >= n + g and q1 + off - 64 j < n + g + l; in the sink iff 64 j + 63 < s.
    int f_lo[3] = {1, 1, 1}, f_hi[3] = {0, 0, 0};
    if (q0 + BQ <= Nq) {
      auto fdiv = [](long long x) -> int { return (int)(x >= 0 ? x / BK : -((-x + BK - 1) / BK)); };
      const long long p0 = (long long)q0 + off, p1 = p0 + BQ - 1;
      const int causal_hi = fdiv(p0 - (BK - 1));
      f_lo[0] = fdiv(p1 - w.n) + 1; f_hi[0] = causal_hi;
      if (w.l > 0) {
        f_lo[1] = fdiv(p1 - ((long long)w.n + w.g + w.l)) + 1;
        f_hi[1] = min(causal_hi, fdiv(p0 - ((long long)w.n + w.g) - (BK - 1)));
      }
      f_lo[2] = 0; f_hi[2] = min(causal_hi, w.s >= BK ? (w.s - BK) / BK : -1);
    }
    // walk of the ranges: tile j steps down to j_last, then the next non-empty range is entered; the
    // current range's bounds live in registers (selects, no indexed local arrays)
    int rr = -1, j = 0, j_last = 0, fl = 1, fh = 0, skip = t0;
    auto next_range = [&]() {
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        if (rr < c && rg[c].hi >= rg[c].lo) {
          if (MERGE && skip > rg[c].hi - rg[c].lo) { skip -= rg[c].hi - rg[c].lo + 1; continue; }
          rr = c; j = rg[c].hi - (MERGE ? skip : 0); j_last = rg[c].lo; fl = f_lo[c]; fh = f_hi[c];
          skip = 0;
          return;
        }
      }
      rr = 3;
    };
    next_range();

    for (int t = 0; t < nt && ok; ++t) {
      const int b_ = NB == 2 ? t & 1 : 0;
      const int k0 = j * BK;
      const bool full = j >= fl && j <= fh;
      const uint32_t t_S = t_lane + b_ * 64;

      ok = mbar_wait(bar_s + b_, (NB == 2 ? t >> 1 : t) & 1, a.status);
      if (!ok) break;
      tc_fence_after();
      uint32_t sr[2][32];
      tmem_ld32(t_S, sr[0]);
      tmem_ld32(t_S + 32, sr[1]);
      tmem_wait_ld();

      if (!full) {
        const int kend = row_valid ? min(rowpos, Nk - 1) : -1;  // last causal key of this row
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          const int base = k0 + c * 32;
          uint32_t mk = interval_bits(rowpos - w.n + 1, kend, base) | interval_bits(0, min(w.s - 1, kend), base);
          if (w.l > 0) mk |= interval_bits(rowpos - (w.n + w.g + w.l) + 1, min(rowpos - (w.n + w.g), kend), base);
#pragma unroll
          for (int e = 0; e < 32; ++e)
            if (!((mk >> e) & 1u)) sr[c][e] = 0xFF800000u;  // -inf
        }
      }
      // row max: four independent chains of 3-input max
      float mxa[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
      for (int c = 0; c < 2; ++c)
#pragma unroll
        for (int e = 0; e < 32; e += 2)
          mxa[(e >> 1) & 3] = max3(mxa[(e >> 1) & 3], __uint_as_float(sr[c][e]), __uint_as_float(sr[c][e + 1]));
      const float mx = fmaxf(fmaxf(mxa[0], mxa[1]), fmaxf(mxa[2], mxa[3])) * a.scale_log2;
      float m_new = m_ref;
      if (mx > m_ref + 8.f) m_new = mx;
      const float alpha = (m_new == m_ref) ? 1.f : ex2(m_ref - m_new);
      const float sub = (m_new == -INFINITY) ? 0.f : m_new;
      m_ref = m_new;
      // rescale the accumulator when some row of this warp moved its reference max
      auto rescale = [&]() {
        if (t > 0 && __any_sync(0xFFFFFFFFu, alpha != 1.f)) {
          const float2 al2 = make_float2(alpha, alpha);
#pragma unroll 1
          for (int c = 0; c < D / 16; ++c) {
            uint32_t ov[16];
            tmem_ld16(t_O + c * 16, ov);
            tmem_wait_ld();
#pragma unroll
            for (int e = 0; e < 16; e += 2) {
              const float2 y = mul2(make_float2(__uint_as_float(ov[e]), __uint_as_float(ov[e + 1])), al2);
              ov[e] = __float_as_uint(y.x); ov[e + 1] = __float_as_uint(y.y);
            }
            tmem_st16(t_O + c * 16, ov);
          }
        }
      };
      if constexpr (NB == 1) rescale();  // S of this step completed behind the product of the step before

      // p = 2^(s * scale - m): packed fp32 pairs for the multiply-add and the row sum
      const float2 nsub2 = make_float2(-sub, -sub);
      float2 rsa[4] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
      uint32_t pk[NB == 2 ? 32 : 16];
#pragma unroll
      for (int c = 0; c < 2; ++c) {
#pragma unroll
        for (int e = 0; e < 32; e += 2) {
          const float2 x = fma2(make_float2(__uint_as_float(sr[c][e]), __uint_as_float(sr[c][e + 1])), sc2, nsub2);
          const float2 pp = make_float2(ex2(x.x), ex2(x.y));
          rsa[(e >> 1) & 3] = add2(rsa[(e >> 1) & 3], pp);
          pk[(NB == 2 ? c * 16 : 0) + e / 2] = pack_bf16(pp.x, pp.y);
        }
        if constexpr (NB == 1) tmem_st16(t_S + c * 16, pk);  // P over the first 32 columns of S
      }
      const float2 rs2 = add2(add2(rsa[0], rsa[1]), add2(rsa[2], rsa[3]));
      l_sum = fmaf(l_sum, alpha, rs2.x + rs2.y);  // (all forms alike, whatever the compiler would merge)

      // Every step waits for the product of the step before (normally long finished): the accumulator
      // may then be rescaled safely, and no thread ever falls two phases behind on this barrier, which
      // its parity wait could not tell apart.
      if (NB == 2 && t > 0) {
        ok = mbar_wait(bar_pv, (t - 1) & 1, a.status);
        if (!ok) break;
        tc_fence_after();
      }
      if constexpr (NB == 2) {
        rescale();
        tmem_st32(t_S, pk);  // P over the first 32 columns of this S buffer
      }
      tmem_wait_st();
      if constexpr (VARLEN) {
        // Last key tile of a packed sequence: the rows after it in shared memory belong to the next sequence.
        // Their P entries are exactly zero, but 0 x (Inf or NaN) in the product would still poison this
        // sequence, so those V rows are cleared before the product may start.
        const int vrows = Nk - j * BK;  // valid rows of this 64-row tile
        if (vrows < BK) {
          ok = mbar_wait(bar_v + (t & 1), (t >> 1) & 1, a.status);
          if (!ok) break;
          uint8_t* vt = sV + (t & 1) * SM::kKV;
          const int nchunk = (BK - vrows) * 8;  // 16-byte chunks per slab
          for (int s_ = 0; s_ < NSLAB; ++s_)
            for (int c_ = r; c_ < nchunk; c_ += 128)
              *reinterpret_cast<uint4*>(vt + s_ * SLAB_K + vrows * 128 + c_ * 16) = make_uint4(0u, 0u, 0u, 0u);
          fence_proxy_async_smem();
        }
      }
      tc_fence_before();
      mbar_arrive(bar_p + b_);
      if (j > j_last) --j; else next_range();
    }

    // ---- epilogue: O / l, LSE ----
    if (nt > 0) ok = mbar_wait(bar_pv, NB == 2 ? (nt - 1) & 1 : 0, a.status) && ok;
    if constexpr (MERGE) {
      // fp32 O goes where this stream's K and V were
      tc_fence_after();
      if (ok && nt > 0) {
#pragma unroll
        for (int c = 0; c < D / 32; ++c) {
          uint32_t ov[32];
          tmem_ld32(t_O + c * 32, ov);
          tmem_wait_ld();
#pragma unroll
          for (int q = 0; q < 8; ++q)
            *reinterpret_cast<uint4*>(sK + r * (D * 4) + (((c * 8 + q) ^ (r & 7)) << 4)) =
                make_uint4(ov[q * 4], ov[q * 4 + 1], ov[q * 4 + 2], ov[q * 4 + 3]);
        }
      }
      reinterpret_cast<float2*>(smem + SM::oState)[stream * BQ + r] = make_float2(m_ref, l_sum);
    } else if (ok && nt > 0) {
      tc_fence_after();
      const float inv = l_sum > 0.f ? 1.f / l_sum : 0.f;
#pragma unroll
      for (int c = 0; c < D / 32; ++c) {
        uint32_t ov[32];
        tmem_ld32(t_O + c * 32, ov);
        tmem_wait_ld();
        // 32 columns = 4 chunks of 8 elements (16 B); slab = (c*32)/64, chunk index within slab
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          uint4 v;
          v.x = pack_bf16(__uint_as_float(ov[q * 8 + 0]) * inv, __uint_as_float(ov[q * 8 + 1]) * inv);
          v.y = pack_bf16(__uint_as_float(ov[q * 8 + 2]) * inv, __uint_as_float(ov[q * 8 + 3]) * inv);
          v.z = pack_bf16(__uint_as_float(ov[q * 8 + 4]) * inv, __uint_as_float(ov[q * 8 + 5]) * inv);
          v.w = pack_bf16(__uint_as_float(ov[q * 8 + 6]) * inv, __uint_as_float(ov[q * 8 + 7]) * inv);
          const int d0 = c * 32 + q * 8;
          const int slab = d0 / 64, chunk = (d0 % 64) / 8;
          if (!tail_rows)
            *reinterpret_cast<uint4*>(sQ + slab * SLAB_Q + tid * 128 + ((chunk ^ (tid & 7)) << 4)) = v;
          else if (row_valid)
            *reinterpret_cast<uint4*>(a.o + ((size_t)h * a.total_q + qbase + row) * D + d0) = v;
        }
      }
      if (row_valid) {
        const size_t li = VARLEN ? (size_t)h * a.total_q + qbase + row : ((size_t)b * a.Hq + h) * Nq + row;
        a.lse[li] = 0.6931471805599453f * (m_ref + log2f(l_sum));
      }
      fence_proxy_async_smem();
    }
    if (!MERGE) asm volatile("bar.sync 1, 128;" ::: "memory");  // the four softmax warps
    if (!MERGE && tid == 0 && ok && nt > 0 && !tail_rows) {
      for (int s = 0; s < NSLAB; ++s) tma_store_4d(&tmO, sQ + s * SLAB_Q, s * 64, qbase + q0, h, bt);
      tma_commit_group();
      tma_wait_group_read<0>();
    }
  }

  if constexpr (MERGE) {
    // Merge of the item's partial states: a cluster's block `rank` writes every csize-th part of the 128 rows.
    if constexpr (SPLIT) cluster_sync();
    else __syncthreads();
    // A thread takes 16 bytes of a row, eight loads of O in flight together with the states that weigh them.  (States first, a
    // thread per row, then O, a part after the other: 4.3 us instead of 1.1 for a cluster of eight.)
    auto merge = [&](auto parts_) {
      constexpr int P = decltype(parts_)::value, U = 8 / P, LPR = D / 4;
      const int per = BQ / csize, first = rank * per;
      const uint32_t aState = smem_u32(smem + SM::oState), aO = smem_u32(smem + SM::oKV);
      auto at = [&](uint32_t addr, int p) { return SPLIT ? map_cluster(addr, p) : addr; };
      for (int i0 = tid; i0 < per * LPR; i0 += kFwdThreads * NS * U) {
        float2 ml[U][P];
        float4 v[U][P];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int i = min(i0 + u * kFwdThreads * NS, per * LPR - 1), r = first + i / LPR, ch = i % LPR;
#pragma unroll
          for (int p = 0; p < P; ++p) {
            ml[u][p] = ld_cluster_f2(at(aState + ((SPLIT ? 0 : p) * BQ + r) * 8, p));
            v[u][p] = make_float4(0.f, 0.f, 0.f, 0.f);
            if (work * p / P < work * (p + 1) / P)  // a part without a step left no O
              v[u][p] = ld_cluster_f4(at(aO + (SPLIT ? 0 : p) * 4 * SM::kKV + r * (D * 4) + ((ch ^ (r & 7)) << 4), p));
          }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int i = i0 + u * kFwdThreads * NS, r = first + i / LPR, ch = i % LPR, row = q0 + r;
          float M = -INFINITY, L = 0.f;
#pragma unroll
          for (int p = 0; p < P; ++p) M = fmaxf(M, ml[u][p].x);
#pragma unroll
          for (int p = 0; p < P; ++p) {
            ml[u][p].x = ml[u][p].x == -INFINITY ? 0.f : ex2(ml[u][p].x - M);
            L = fmaf(ml[u][p].y, ml[u][p].x, L);
          }
          const float inv = L == 0.f ? 0.f : 1.f / L;  // a NaN sum has to come out as NaN
          float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
          for (int p = 0; p < P; ++p) {
            const float wgt = ml[u][p].x * inv;
            o.x = fmaf(v[u][p].x, wgt, o.x); o.y = fmaf(v[u][p].y, wgt, o.y);
            o.z = fmaf(v[u][p].z, wgt, o.z); o.w = fmaf(v[u][p].w, wgt, o.w);
          }
          if (i < per * LPR && row < Nq) {
            __nv_bfloat16* dst = a.o + (VARLEN ? ((size_t)h * a.total_q + qbase + row) * D
                                               : (size_t)b * a.so.b + (size_t)h * a.so.h + (size_t)row * a.so.t);
            *reinterpret_cast<uint2*>(dst + ch * 4) = make_uint2(pack_bf16(o.x, o.y), pack_bf16(o.z, o.w));
            if (ch == 0) {
              const size_t li = VARLEN ? (size_t)h * a.total_q + qbase + row : ((size_t)b * a.Hq + h) * Nq + row;
              a.lse[li] = 0.6931471805599453f * (M + log2f(L));
            }
          }
        }
      }
    };
    if (work > 0) {
      if constexpr (!SPLIT) merge(std::integral_constant<int, NS>());
      else if (csize == 2) merge(std::integral_constant<int, 2>());
      else if (csize == 4) merge(std::integral_constant<int, 4>());
      else merge(std::integral_constant<int, 8>());
    }
    if constexpr (SPLIT) cluster_sync();  // no block leaves while another one reads its shared memory
  }

  // ---- teardown ----
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    __syncwarp();
    tmem_dealloc(*tmem_holder, TMEM_COLS);
  }
}

// One launch for both layouts.  Batched: cu_q == nullptr, tensors [B,H,N,D].  Packed: tensors
// [H,total,D]; the grid is sized from total_q / BQ + B, an upper bound of the batch's tile count.
template <int D, bool VARLEN>
int launch_fwd(const void* q, const void* k, const void* v, void* o, float* lse, int B, int Nq, int Nk, int Hq,
               int Hkv, const cowa_params_t* p, const CowaHeadWindows& hw, const int* cu_q, const int* cu_k,
               int total_q, int total_k, cudaStream_t st) {
  CUtensorMap mq, mk, mv, mo;
  int rc;
  const int rows_q = VARLEN ? total_q : Nq, rows_k = VARLEN ? total_k : Nk;
  const int nb = VARLEN ? 1 : B;  // packed tensors are [H, total, D]
  CowaStrides sq, sk, sv, so;
  if (VARLEN && cowa::any_stride_set(p)) return COWA_ERR_UNSUPPORTED;
  if ((rc = cowa::resolve_strides(p->q_strides, Hq, rows_q, D, &sq))) return rc;
  if ((rc = cowa::resolve_strides(p->k_strides, Hkv, rows_k, D, &sk))) return rc;
  if ((rc = cowa::resolve_strides(p->v_strides, Hkv, rows_k, D, &sv))) return rc;
  if ((rc = cowa::resolve_strides(p->o_strides, Hq, rows_q, D, &so))) return rc;
  if ((rc = cowa::make_tensor_map(&mq, q, cowa::MapType::BF16, D, rows_q, Hq, nb, sq, 64, BQ))) return rc;
  if ((rc = cowa::make_tensor_map(&mk, k, cowa::MapType::BF16, D, rows_k, Hkv, nb, sk, 64, BK))) return rc;
  if ((rc = cowa::make_tensor_map(&mv, v, cowa::MapType::BF16, D, rows_k, Hkv, nb, sv, 64, BK))) return rc;
  if ((rc = cowa::make_tensor_map(&mo, o, cowa::MapType::BF16, D, rows_q, Hq, nb, so, 64, BQ))) return rc;
  FwdArgs a;
  a.lse = lse;
  a.status = cowa::device_status_word();
  if (!a.status) return COWA_ERR_CUDA;
  a.B = B; a.Nq = Nq; a.Nk = Nk; a.Hq = Hq; a.Hkv = Hkv; a.G = Hq / Hkv;
  a.scale_log2 = p->softmax_scale * 1.4426950408889634f;
  a.wins = hw;
  a.cu_q = cu_q; a.cu_k = cu_k; a.o = static_cast<__nv_bfloat16*>(o); a.total_q = total_q; a.total_k = total_k; a.so = so;
  a.sink = p->sink; a.local = p->local;
  a.hkv_global = p->hkv_global > 0 ? p->hkv_global : Hkv;
  a.hkv_offset = p->hkv_offset; a.full_attn = p->full_attn; a.explicit_windows = p->windows != nullptr;
  const long long tiles = VARLEN ? (long long)total_q / BQ + B : (long long)((Nq + BQ - 1) / BQ) * B;
  const int qn = VARLEN ? std::max(total_q / B, 1) : Nq, kn = VARLEN ? std::max(total_k / B, 1) : Nk;
  int keys = 0;  // visited by the longest list, tile remainders included
  for (int h = 0; h < Hkv; ++h) {
    CowaWin w = hw.w[h];
    if (VARLEN && p->full_attn) w.n = kn;
    else if (VARLEN && !p->windows) w = cowa_default_window(kn, a.hkv_global, a.hkv_offset + h, a.sink, a.local);
    const long long width = (long long)std::min(w.s, kn) + std::min(w.n, kn) + std::min(w.l, kn) + 2 * BQ;
    keys = std::max(keys, (int)std::min<long long>(width, kn));
  }
  // Packed batches: order of the items.  By length where the average sequence has 1024 keys to visit, or where the blocks of
  // single heads make four waves at most and a long list among the last ones shows (20 prompts of 30 to 1000 tokens, 4 heads:
  // 33 us, 38 in the batch's order; 7 of 4292 tokens, 16 heads: 46, 54).  Else lists are over so soon that finding an item by
  // its length costs more than it gives (30 prompts of 100 tokens, 32 heads, D = 64: 24 us, 21 in the batch's order).
  a.longest_first = VARLEN && B <= kLongestFirst && (keys >= 1024 || tiles * Hq <= 8 * cowa::sm_count());
  // The one-head kernel's forms, judged for packed batches by their average sequence, so that equal lengths give what the
  // batched call gives, bit for bit.
  const int sms = cowa::sm_count(), steps = (keys + BK - 1) / BK;
  const long long blocks = tiles * Hq, heads = (long long)((qn + BQ - 1) / BQ) * B * Hq;
  if (blocks > 0x7FFFFFFFll) return COWA_ERR_UNSUPPORTED;
  // Clusters while blocks of half the items do not fill the SMs' two places each: a short list has too little to share for a
  // second block per SM (us, clusters of 1 / 2 / 4 / 8, D = 64: 32 items of 12 steps 13.5 / 10.6 / 8.2 / 9.3, of 164 steps
  // 165 / 71 / 38 / 29; 56 of 28 28 / 17 / 14.3 / 20; 8 of 14 17.7 / 11.6 / 8.7 / 7.0; D = 128: 32 of 12 12.7 / 12.7 / 10.6 /
  // 12.5, 56 of 28 27 / 20 / 18 / 25, 8 of 14 20 / 15 / 11 / 9).  At D = 128 they are also better than the pair kernel's, whose
  // items are half as many, where lists differ in length (128 items of up to 42 steps 26 / 33; 512 tokens behind 32K 59 / 55).
  // More items at D = 64, one block of one buffer / four streams / one block of two buffers, us:
  //   128 items of 20 steps   22 / 15 / 19    192 of 10   21.5 / 21 / 18.5   256 of 12   20 / 25 / 18.5   288 of 9   22 / 29 / 21
  //   160 of 14               17 / 14 / 15    192 of 19   51 / 28 / 42       256 of 64   54 / 31 / 45     288 of 43  57 / 42 / 48
  //   320 of up to 12         19 / 26 / 18    352 of 14   46 / 45 / 39       384 of 52   125 / 77 / 105   320 of 40  36 / 33 / 31
  //   352 of 16, all alike    32 / 38 / 36    448 alike   35 / 47 / 39       576 of 17   28 / 42 / 32     696 of 95  132 / 112
  // Streams shorten the longest list but leave one block per SM; two buffers shorten a block's step where two or three blocks
  // are all an SM gets; one buffer wins as soon as four have work to the end: lists alike, or more of them.  (Streams from the
  // line on also where all lists are alike, 192 of 22 steps 30 / 30 / 27: an average of packed lengths does not tell.)
  const bool alike = kn >= 2ll * qn;  // every tile's list is about as long
  int streams = 1, split = 1;
  [[maybe_unused]] bool deep = false;  // two S buffers, at D = 64
  if (4 * heads <= 2 * sms) {
    while (split < 8 && 2 * split * heads <= (steps >= 24 ? 2 * sms : sms) && 2 * split <= steps) split *= 2;
    // A merge is as long as four steps, six at D = 128 (the other blocks' O comes in twice as many pieces), and longer where clusters
    // of four have to share SMs, as they lie within one GPC each: a list that is cut has to save at least that many.  us, one block / the
    // clusters above: D = 64, 16 items of 2 steps 4.5 / 6.5, 4 6.0 / 6.3, 5 6.7 / 6.8, 6 7.5 / 6.9, 48 of 6 7.6 / 8.1, 8 9.2 / 9.0;
    // D = 128, 16 of 2 5.3 / 8.5, 4 6.8 / 7.8, 6 8.3 / 8.5, 8 9.8 / 10.0, 10 11.4 / 10.6, 48 of 8 10.0 / 11.4, 12 13.1 / 13.0, 36 of 8 10.0 / 11.1,
    // 10 11.5 / 12.0, 12 13.0 / 12.3.
    const bool crowded = split == 4 && 9 * split * heads > 8ll * sms;
    if (steps - steps / split < (D == 64 ? (crowded ? 6 : 4) : (crowded ? 9 : 6))) split = 1;
    deep = split == 1;  // (one block on an SM)
  } else if (D == 64) {
    if (heads <= 2 * sms ? 12 * steps > heads : heads <= 3 * sms ? 8 * steps > heads : heads <= 5 * sms && steps >= 64) streams = 4;
    else deep = heads <= (alike && !VARLEN ? 2 : 3) * sms;  // (the same sums in the same order as with one buffer)
  } else if (heads <= sms && steps >= 32 && (!alike || a.G % 2)) {
    split = 2;
  }
  if (D == 128 && split == 1 && a.G % 2 == 0) {
    // Which kernel (us, one-head / pair kernel; at D = 64 the exponentials bound both, and the one-head kernel keeps them
    // busier):
    //   No more items than clusters of two that the device holds, and a list long enough to pay for the merge: two blocks share
    //     an item.  Hq 32, Hkv 8, Nq 128: 1816 keys 37.9 / 25.6 (fewer items: the clusters above).
    //   Else the pair kernel pays when its larger items still share out evenly (the figures are from a fixed share of the
    //   items per block; now that blocks take items as they come free it has gained up to a fifth where the rule takes it,
    //   and the lines have been left where they are):
    //     every tile's list is about as long (a chunk behind a cache of its own length or more) and not short: Hq 32,
    //     Nq 1024, 1129 keys 1.00, 1816 keys 1.09, 4941 keys 1.13 times the one-head kernel's rate;
    //     causal lists from nothing up: three items per SM, or half of that and lists of 1280 keys.  T 2048, Hq 16, local
    //     1024 (0.9 items per SM) 0.88 times; Hq 32 (1.7) local 128 0.87, local 1024 1.13; T 3072 (2.6) local 128 0.91,
    //     local 2048 1.10; T 8192 (6.9) local 1024 1.03; T 32768, local 2048 1.13.  In between the last round decides, by
    //     up to a tenth either way (T 6000, Hq 16, 2.5 items per SM: 0.90; T 2048, Hq 32, 1.7: 1.13).
    const long long items = tiles * (Hq / 2), judged = (long long)((qn + BQ - 1) / BQ) * B * (Hq / 2);
    if (items > 0x7FFFFFFFll) return COWA_ERR_UNSUPPORTED;
    const bool shared = judged <= cowa::resident_pairs();
    const bool rounds = judged >= 3 * cowa::sm_count() || (alike ? keys >= 1536 : keys >= 1280 && 2 * judged >= 3 * cowa::sm_count());
    // Packed batches whose average sequence has fewer than 1024 keys to visit: three quarters of the items that there are at
    // least in fixed shares, the rest taken over (cowa_fwd_pair.cu).  Half is 2 to 4 % slower for equal lengths, nine tenths
    // 17 % for 24 of 60 to 7000 tokens, local 128; from 1024 keys on lists hide what taking over costs.
    const int share = VARLEN && keys < 1024 ? (int)(0.75 * (total_q / BQ) * (Hq / 2) / cowa::sm_count()) : 1;
    if (shared ? keys >= 1536 : rounds)
      return cowa::launch_fwd_pair<128, VARLEN>(mq, mk, mv, mo, a, items, std::max(share, 1), shared ? 2 : 1, st);
  }
  auto launch = [&](auto kernel, int smem) -> int {
    COWA_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(blocks * split)); cfg.blockDim = dim3(kFwdThreads * streams); cfg.dynamicSmemBytes = smem; cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = (unsigned)split; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr; cfg.numAttrs = split > 1 ? 2 : 1;
    COWA_CUDA_TRY(cudaLaunchKernelEx(&cfg, kernel, mq, mk, mv, mo, a));
    return COWA_OK;
  };
  if (split > 1) return launch(cowa_fwd_kernel<D, VARLEN, 2, 1, true>, FwdSmem<D, 1, true>::kBytes);
  if constexpr (D == 64) {
    if (streams > 1) return launch(cowa_fwd_kernel<D, VARLEN, 1, 4, false>, FwdSmem<D, 4, false>::kBytes);
    if (!deep) return launch(cowa_fwd_kernel<D, VARLEN, 1, 1, false>, FwdSmem<D, 1, false>::kBytes);
  }
  return launch(cowa_fwd_kernel<D, VARLEN, 2, 1, false>, FwdSmem<D, 1, false>::kBytes);
}

}  // namespace

extern "C" {

int cowa_prefill(const void* q, const void* k, const void* v, void* o, float* lse, int B, int Nq, int Nk, int Hq,
                 int Hkv, int D, const cowa_params_t* p, void* stream) {
  if (!q || !k || !v || !o || !lse || !p) return COWA_ERR_INVALID_ARG;
  if (B <= 0 || Nq <= 0 || Nk < Nq || Hq <= 0 || Hkv <= 0 || Hq % Hkv != 0) return COWA_ERR_INVALID_ARG;
  if (!(p->softmax_scale > 0.f)) return COWA_ERR_INVALID_ARG;
  if (D != 64 && D != 128) return COWA_ERR_UNSUPPORTED;
  if (!cowa::aligned16(q) || !cowa::aligned16(k) || !cowa::aligned16(v) || !cowa::aligned16(o))
    return COWA_ERR_MISALIGNED;
  CowaHeadWindows hw;
  int rc = cowa::resolve_windows(Nk, Hkv, p, &hw);
  if (rc != COWA_OK) return rc;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  return D == 128 ? launch_fwd<128, false>(q, k, v, o, lse, B, Nq, Nk, Hq, Hkv, p, hw, nullptr, nullptr, 0, 0, st)
                  : launch_fwd<64, false>(q, k, v, o, lse, B, Nq, Nk, Hq, Hkv, p, hw, nullptr, nullptr, 0, 0, st);
}

int cowa_prefill_varlen(const void* q, const void* k, const void* v, void* o, float* lse, const int32_t* cu_seqlens_q,
                        const int32_t* cu_seqlens_k, int B, int total_q, int total_k, int Hq, int Hkv, int D,
                        const cowa_params_t* p, void* stream) {
  if (!q || !k || !v || !o || !lse || !p || !cu_seqlens_q || !cu_seqlens_k) return COWA_ERR_INVALID_ARG;
  if (B <= 0 || total_q <= 0 || total_k < total_q || Hq <= 0 || Hkv <= 0 || Hq % Hkv != 0)
    return COWA_ERR_INVALID_ARG;
  if (!(p->softmax_scale > 0.f)) return COWA_ERR_INVALID_ARG;
  if (D != 64 && D != 128) return COWA_ERR_UNSUPPORTED;
  if (!cowa::aligned16(q) || !cowa::aligned16(k) || !cowa::aligned16(v) || !cowa::aligned16(o))
    return COWA_ERR_MISALIGNED;
  // Explicit tuples are validated and copied here; the default rule is evaluated per sequence on the
  // device (any positive N_k passes the same checks on sink / local / head offsets).
  CowaHeadWindows hw;
  int rc = cowa::resolve_windows(total_k, Hkv, p, &hw);
  if (rc != COWA_OK) return rc;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  return D == 128 ? launch_fwd<128, true>(q, k, v, o, lse, B, 0, 0, Hq, Hkv, p, hw, cu_seqlens_q,
                                          cu_seqlens_k, total_q, total_k, st)
                  : launch_fwd<64, true>(q, k, v, o, lse, B, 0, 0, Hq, Hkv, p, hw, cu_seqlens_q,
                                         cu_seqlens_k, total_q, total_k, st);
}

int cowa_fwd(const void* q, const void* k, const void* v, void* o, float* lse, int B, int T, int Hq, int Hkv, int D,
             const cowa_params_t* p, void* stream) {
  return cowa_prefill(q, k, v, o, lse, B, T, T, Hq, Hkv, D, p, stream);
}

}  // extern "C"
