// Split-KV single-token decode for CoWindow Attention (Sec. 2.3 "Decoding"): the forward
// with N_q = 1, delta = N_k - 1 - i_k, windows recomputed from the current key length of each
// sequence; the visible rows of a head are divided over split programs whose partial
// online-softmax states are merged afterwards.
//
// HBM-bound: every visible K and V row is read exactly once, with 128-bit loads, straight
// into registers.  Per (sequence, KV head, split) one 128-thread block, 5 blocks per SM:
//   1. scores:  each warp takes 16 visible rows at a time; K rows are loaded as the A
//      fragment of mma.sync m16n8k16 (bf16, fp32 accumulate), the group's query vectors are
//      the B fragment.  The contraction index is permuted identically on both operands so
//      that every thread's loads are 16-byte vectors.  Scores (log2 units) go to shared memory.
//   2. block-wide max / exp2 / sum per QO head (no running rescale: the split's scores are
//      all in shared memory before any V row is touched).
//   3. values:  again mma.sync m16n8k16, O^T += V^T P^T with 16 visible rows per instruction; V rows are
//      loaded with 16-byte vectors and neighbouring rows are paired with byte permutes (the d index is
//      permuted inside the fragment and restored on output); the four warps' partial sums meet in shared
//      memory; un-normalised partial (o, m, l) written to the workspace.
// A second kernel merges the splits (log-sum-exp combine with warp shuffles).
#include <cuda_bf16.h>

#include <algorithm>

#include "cowa_common.h"
#include "cowa_ptx.cuh"

namespace {

constexpr int kThreads = 128;
constexpr int kChunkCap = 1024;  // max visible rows per split (scores of a split live in shared memory)
constexpr int kScStride = kChunkCap + 8;  // row stride of the score array: heads land in different banks

// Scratch of cowa_decode_static: lives in the library's device image, so every GPU that loads the
// library keeps these bytes reserved until the process exits.
constexpr size_t kStaticScratchBytes = 8u << 20;
static __device__ __align__(256) unsigned char g_decode_static_scratch[kStaticScratchBytes];

// Device address of the scratch array on the current device.  The array's name is only a
// host-side handle here; the address the kernels need comes from cudaGetSymbolAddress, looked
// up once per device with that device current.
void* static_scratch_ptr(cudaError_t* err) {
  static void* cache[64] = {nullptr};
  int dev = 0;
  *err = cudaGetDevice(&dev);
  if (*err != cudaSuccess) return nullptr;
  if (dev < 0 || dev >= 64) { *err = cudaErrorInvalidDevice; return nullptr; }
  if (!cache[dev]) {
    void* ptr = nullptr;
    *err = cudaGetSymbolAddress(&ptr, g_decode_static_scratch);
    if (*err != cudaSuccess) return nullptr;
    cache[dev] = ptr;
  }
  return cache[dev];
}

struct DecodeArgs {
  const __nv_bfloat16* q;
  const __nv_bfloat16* kc;
  const __nv_bfloat16* vc;
  const int32_t* lens;
  float* ws_o;  // [B, Hq, S, D]
  float* ws_m;  // [B, Hq, S]
  float* ws_l;
  int B, Tmax, Hq, Hkv;
  int S;      // splits of a (sequence, KV head)
  int ahead;  // V is prefetched: splits of at most 2 * kThreads rows
  CowaStrides sk, sv;  // element strides (batch, head, token) of the contiguous-row cache
  int sink, near, hkv_global, hkv_offset, full_attn;
  float scale_log2;
};

// Position of the v-th visible row (v in the concatenation of the head's ranges).
struct VisMap {
  int lo0, n0, lo1, n1, lo2;
  __device__ __forceinline__ int token(int v) const {
    return v < n0 ? lo0 + v : (v < n0 + n1 ? lo1 + (v - n0) : lo2 + (v - n0 - n1));
  }
};

__device__ __forceinline__ void mma_bf16_16816(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2,
                                               uint32_t a3, uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};\n"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

__device__ __forceinline__ uint4 ldg128(const void* p) {
  uint4 r;
  asm volatile("ld.global.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w)
               : "l"(p));
  return r;
}

// G = columns of the mma n-tile in use: the query heads of the group.
template <int D, int G>
// 5 blocks per SM (up to 102 registers, no spills) measured best: fewer, longer splits than at 7 per SM
// (D = 64, groups below 8: 7)
__global__ void __launch_bounds__(kThreads, D == 64 && G < 8 ? 7 : 5) cowa_decode_split_kernel(const DecodeArgs a) {
  static_assert(D == 64 || D == 128, "head dim");
  static_assert(G >= 1 && G <= 8, "group size per mma n-tile");
  constexpr int KC = D / 32;          // 32-wide d chunks (two k16 steps each)

  __shared__ __align__(16) float sc[G * kScStride];  // scores, later the value-phase reduction buffer
  __shared__ float m_s[G], l_s[G];

  cowa_ptx::grid_enter();  // the merge kernel's blocks may be scheduled beside this one's; they wait for its results
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int split = blockIdx.x, hk = blockIdx.y, b = blockIdx.z, S = a.S;
  const size_t state = ((size_t)(b * a.Hkv + hk) * G) * S + split;  // of the first head, head c's is at state + c * S
  const int Nk = a.lens[b];

  // visible ranges of this head for the current key length
  CowaWin w;
  if (a.full_attn) { w.s = 0; w.n = Nk; w.g = 0; w.l = 0; }
  else w = cowa_default_window(Nk, a.hkv_global, a.hkv_offset + hk, a.sink, a.near);
  CowaRange rg[3];
  const int nr = cowa_decode_ranges(w, Nk, rg);
  // index of column c in q ([B, Hq] order)
  auto col = [&](int c) -> size_t { return (size_t)b * a.Hq + (size_t)hk * G + c; };
  // address of cache row `tok` of this (sequence, KV head)
  auto row_ptr = [&](const __nv_bfloat16* base, const CowaStrides& cs, int tok) -> const __nv_bfloat16* {
    return base + (size_t)b * cs.b + (size_t)hk * cs.h + (size_t)tok * cs.t;
  };
  VisMap vm;
  vm.lo0 = rg[0].lo; vm.n0 = nr > 0 ? rg[0].hi - rg[0].lo + 1 : 0;
  vm.lo1 = nr > 1 ? rg[1].lo : 0; vm.n1 = nr > 1 ? rg[1].hi - rg[1].lo + 1 : 0;
  vm.lo2 = nr > 2 ? rg[2].lo : 0;
  const int n2 = nr > 2 ? rg[2].hi - rg[2].lo + 1 : 0;
  const int V = vm.n0 + vm.n1 + n2;

  // From this sequence's length and the call's sizes alone: its result does not depend on how long the others are.
  const int chunk = ((V + S - 1) / S + 15) & ~15;
  const int c0 = split * chunk;
  const int clen = min(chunk, V - c0);  // <= kChunkCap by the host's choice of S

  if (clen <= 0) {  // empty split: neutral partial state
    for (int i = tid; i < G * D; i += kThreads) a.ws_o[(state + (size_t)(i / D) * S) * D + i % D] = 0.f;
    if (tid < G) {
      a.ws_m[state + tid * S] = -INFINITY;
      a.ws_l[state + tid * S] = 0.f;
    }
    return;
  }
  // Small calls: V is on its way to L2 while K is read and weighed (8K of context, one sequence 8.8 us, so 8.4).  Where bandwidth
  // counts, K would wait behind it, and it comes out of L2 a second time (8 sequences, 8 heads of 2000 rows, 65 MB: 16.5 us, so 18.3).
  if (a.ahead) {
#pragma unroll
    for (int r = tid; r < 2 * kThreads; r += kThreads)
      if (r < clen) {
        const char* row = reinterpret_cast<const char*>(row_ptr(a.vc, a.sv, vm.token(c0 + r)));
#pragma unroll
        for (int i = 0; i < D * 2; i += 128) asm volatile("prefetch.global.L2 [%0];" ::"l"(row + i));
      }
  }

  // ---------------- phase 1: scores ----------------
  {
    const int g = lane >> 2, t = lane & 3;
    // B fragments: query head g (zero beyond the group), permuted contraction index
    uint32_t bq[KC][4];
#pragma unroll
    for (int cc = 0; cc < KC; ++cc) {
      uint4 x = make_uint4(0, 0, 0, 0);
      if (g < G) x = *reinterpret_cast<const uint4*>(a.q + col(g) * D + cc * 32 + t * 8);
      bq[cc][0] = x.x; bq[cc][1] = x.y; bq[cc][2] = x.z; bq[cc][3] = x.w;
    }
    const int nblk = (clen + 15) >> 4;
    for (int blk = warp; blk < nblk; blk += kThreads / 32) {
      const int rA = blk * 16 + g, rB = rA + 8;
      const int tokA = vm.token(c0 + min(rA, clen - 1));
      const int tokB = vm.token(c0 + min(rB, clen - 1));
      const __nv_bfloat16* pa = row_ptr(a.kc, a.sk, tokA) + t * 8;
      const __nv_bfloat16* pb = row_ptr(a.kc, a.sk, tokB) + t * 8;
      uint4 ka[KC], kb[KC];
#pragma unroll
      for (int cc = 0; cc < KC; ++cc) { ka[cc] = ldg128(pa + cc * 32); kb[cc] = ldg128(pb + cc * 32); }
      float c[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int cc = 0; cc < KC; ++cc) {
        mma_bf16_16816(c, ka[cc].x, kb[cc].x, ka[cc].y, kb[cc].y, bq[cc][0], bq[cc][1]);
        mma_bf16_16816(c, ka[cc].z, kb[cc].z, ka[cc].w, kb[cc].w, bq[cc][2], bq[cc][3]);
      }
      // c[0],c[1]: row rA, heads 2t, 2t+1;  c[2],c[3]: row rB
      const int h0 = 2 * t, h1 = 2 * t + 1;
      if (rA < clen) {
        if (h0 < G) sc[h0 * kScStride + rA] = c[0] * a.scale_log2;
        if (h1 < G) sc[h1 * kScStride + rA] = c[1] * a.scale_log2;
      }
      if (rB < clen) {
        if (h0 < G) sc[h0 * kScStride + rB] = c[2] * a.scale_log2;
        if (h1 < G) sc[h1 * kScStride + rB] = c[3] * a.scale_log2;
      }
    }
  }
  __syncthreads();

  // ---------------- phase 2: max, exp2, sum per head ----------------
  for (int h = warp; h < G; h += kThreads / 32) {
    float* s = sc + h * kScStride;
    float m = -INFINITY;
    for (int r = lane; r < clen; r += 32) m = fmaxf(m, s[r]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    float l = 0.f;
    for (int r = lane; r < clen; r += 32) {
      float p = exp2f(s[r] - m);
      s[r] = p;
      l += p;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
    if (lane == 0) { m_s[h] = m; l_s[h] = l; }
  }
  __syncthreads();

  // ---------------- phase 3: values, O^T[d, h] += V^T[d, rows] P^T[rows, h] on the tensor cores ----------------
  // 16 visible rows per mma.  A = V^T: thread (g, t) loads 16 bytes (8 consecutive d) of rows 2t, 2t+1, 2t+8,
  // 2t+9 and pairs equal d of neighbouring rows with byte permutes; the row index of an m-tile is a
  // permutation of d (row g <-> d = 8g + 2i, row g+8 <-> d = 8g + 2i + 1 for m-tile i), undone when the
  // accumulators are written out.  B = P^T (bf16), head g of the group in column g.
  {
    const int g = lane >> 2, t = lane & 3;
    constexpr int NB = D / 64;
    float acc[NB][4][4];
#pragma unroll
    for (int bb = 0; bb < NB; ++bb)
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[bb][i][c] = 0.f;
    const int nblk = (clen + 15) >> 4;
    for (int blk = warp; blk < nblk; blk += kThreads / 32) {
      const int r0 = blk * 16 + 2 * t;
      const int rr[4] = {r0, r0 + 1, r0 + 8, r0 + 9};
      uint4 vv[4][NB];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const __nv_bfloat16* src = row_ptr(a.vc, a.sv, vm.token(c0 + min(rr[k], clen - 1))) + g * 8;
#pragma unroll
        for (int bb = 0; bb < NB; ++bb) vv[k][bb] = ldg128(src + bb * 64);
      }
      float pr[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) pr[k] = (g < G && rr[k] < clen) ? sc[g * kScStride + rr[k]] : 0.f;
      uint32_t b0, b1;
      asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(b0) : "f"(pr[1]), "f"(pr[0]));
      asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(b1) : "f"(pr[3]), "f"(pr[2]));
#pragma unroll
      for (int bb = 0; bb < NB; ++bb) {
        const uint32_t x0[4] = {vv[0][bb].x, vv[0][bb].y, vv[0][bb].z, vv[0][bb].w};
        const uint32_t x1[4] = {vv[1][bb].x, vv[1][bb].y, vv[1][bb].z, vv[1][bb].w};
        const uint32_t x2[4] = {vv[2][bb].x, vv[2][bb].y, vv[2][bb].z, vv[2][bb].w};
        const uint32_t x3[4] = {vv[3][bb].x, vv[3][bb].y, vv[3][bb].z, vv[3][bb].w};
#pragma unroll
        for (int i = 0; i < 4; ++i)
          mma_bf16_16816(acc[bb][i], __byte_perm(x0[i], x1[i], 0x5410), __byte_perm(x0[i], x1[i], 0x7632),
                         __byte_perm(x2[i], x3[i], 0x5410), __byte_perm(x2[i], x3[i], 0x7632), b0, b1);
      }
    }
    __syncthreads();  // scores no longer needed: reuse their space as red[warp][h][d]
    static_assert((kThreads / 32) * D <= kChunkCap, "reduction buffer fits the score buffer");
#pragma unroll
    for (int bb = 0; bb < NB; ++bb)
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int d = bb * 64 + 8 * g + 2 * i;
        const int h0 = 2 * t, h1 = 2 * t + 1;
        if (h0 < G) *reinterpret_cast<float2*>(sc + ((size_t)(warp * G + h0) * D + d)) = make_float2(acc[bb][i][0], acc[bb][i][2]);
        if (h1 < G) *reinterpret_cast<float2*>(sc + ((size_t)(warp * G + h1) * D + d)) = make_float2(acc[bb][i][1], acc[bb][i][3]);
      }
  }
  __syncthreads();
  for (int i = tid; i < G * D; i += kThreads) {
    float s = 0.f;
#pragma unroll
    for (int r = 0; r < kThreads / 32; ++r) s += sc[r * G * D + i];
    a.ws_o[(state + (size_t)(i / D) * S) * D + i % D] = s;
  }
  if (tid < G) {
    a.ws_m[state + tid * S] = m_s[tid];
    a.ws_l[state + tid * S] = l_s[tid];
  }
}

// Merge of the split states: M = max m_s, L = sum l_s 2^(m_s - M), o = sum o_s 2^(m_s - M) / L,
// lse = ln2 * (M + log2 L).  One block per (sequence, QO head).  A warp takes every W-th split, eight at a time, D/32 columns per
// lane, states and O in one round trip, and the running maximum moves between such groups; the warps' results meet in shared memory.
// W: sixteen warps (one sequence of 57 700 visible rows in 452 splits: with four 16 us of 29 were this kernel); four are enough up
// to 32 splits, where a lane reads one split's state and every warp knows M and L.  That form has 32 registers, so that its
// blocks wait beside five of the split kernel's (with 72: 8 sequences of 8000 tokens 16.6 us, so 17.1; held to 32 with spills
// 17.9).
template <int D, int W>
__global__ void __launch_bounds__(W * 32) cowa_decode_combine_kernel(const DecodeArgs a, __nv_bfloat16* o, float* lse) {
  constexpr int V = D / 32, U = 8;  // columns per lane, splits of a group
  constexpr bool kOnce = W * U == 32;  // S <= 32
  __shared__ float part[W][D], part_m[W], part_l[W];
  const int bh = blockIdx.x;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int S = a.S;
  const size_t first = (size_t)bh * S;
  cowa_ptx::grid_enter();
  const float* m = a.ws_m + first;
  const float* l = a.ws_l + first;
  const float* po = a.ws_o + first * D + lane * V;
  float mx = -INFINITY, L = 0.f, acc[V];
#pragma unroll
  for (int i = 0; i < V; ++i) acc[i] = 0.f;
  if constexpr (kOnce) {
    const float ms = lane < S ? m[lane] : -INFINITY;
    const float ls = lane < S ? l[lane] : 0.f;
    float x[U][V];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int s = warp + W * u;
#pragma unroll
      for (int i = 0; i < V; ++i) x[u][i] = s < S ? po[(size_t)s * D + i] : 0.f;
    }
    mx = ms;
#pragma unroll
    for (int k = 16; k > 0; k >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, k));
    const float w = exp2f(ms - mx);  // empty splits: m = -inf -> weight 0
    L = ls * w;
#pragma unroll
    for (int k = 16; k > 0; k >>= 1) L += __shfl_xor_sync(0xffffffffu, L, k);
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const float wu = __shfl_sync(0xffffffffu, w, (warp + W * u) & 31);
#pragma unroll
      for (int i = 0; i < V; ++i) acc[i] = fmaf(x[u][i], wu, acc[i]);
    }
  } else {
    for (int s0 = warp; s0 < S; s0 += W * U) {
      const bool in = lane < U && s0 + lane * W < S;
      const float ms = in ? m[s0 + lane * W] : -INFINITY;
      const float ls = in ? l[s0 + lane * W] : 0.f;
      float x[U][V];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int s = s0 + u * W;
        const float* src = po + (size_t)s * D;
        if constexpr (V == 4) {
          const float4 y = s < S ? *reinterpret_cast<const float4*>(src) : make_float4(0.f, 0.f, 0.f, 0.f);
          x[u][0] = y.x; x[u][1] = y.y; x[u][2] = y.z; x[u][3] = y.w;
        } else {
          const float2 y = s < S ? *reinterpret_cast<const float2*>(src) : make_float2(0.f, 0.f);
          x[u][0] = y.x; x[u][1] = y.y;
        }
      }
      float top = ms;
#pragma unroll
      for (int k = U / 2; k > 0; k >>= 1) top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, k));
      top = fmaxf(__shfl_sync(0xffffffffu, top, 0), mx);
      const float old = mx == -INFINITY ? 0.f : exp2f(mx - top), w = ms == -INFINITY ? 0.f : exp2f(ms - top);
      mx = top;
      float sum = ls * w;
#pragma unroll
      for (int k = U / 2; k > 0; k >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, k);
      L = L * old + __shfl_sync(0xffffffffu, sum, 0);
#pragma unroll
      for (int i = 0; i < V; ++i) acc[i] *= old;
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const float wu = __shfl_sync(0xffffffffu, w, u);
#pragma unroll
        for (int i = 0; i < V; ++i) acc[i] = fmaf(x[u][i], wu, acc[i]);
      }
    }
    if (lane == 0) { part_m[warp] = mx; part_l[warp] = L; }
  }
#pragma unroll
  for (int i = 0; i < V; ++i) part[warp][lane * V + i] = acc[i];
  __syncthreads();
  if (tid < D) {
    float v;
    if constexpr (kOnce) {
      v = (part[0][tid] + part[1][tid]) + (part[2][tid] + part[3][tid]);
    } else {
      mx = part_m[0];
#pragma unroll
      for (int k = 1; k < W; ++k) mx = fmaxf(mx, part_m[k]);
      L = v = 0.f;
#pragma unroll
      for (int k = 0; k < W; ++k) {
        const float w = part_m[k] == -INFINITY ? 0.f : exp2f(part_m[k] - mx);
        L = fmaf(part_l[k], w, L);
        v = fmaf(part[k][tid], w, v);
      }
    }
    o[(size_t)bh * D + tid] = __float2bfloat16_rn(v / L);
    if (lse && tid == 0) lse[bh] = 0.6931471805599453f * (mx + log2f(L));
  }
}

// Upper bound of visible rows per head for any key length <= Tmax.
int max_visible(int Tmax, int hg, const cowa_params_t* p) {
  if (p->full_attn) return Tmax;
  long long shared = (long long)p->sink + p->local;
  if (shared >= Tmax) return Tmax;
  long long band = ((long long)Tmax - shared + hg - 1) / hg;  // widest band, ceil(L / Hk)
  long long v = shared + band;
  return (int)(v < Tmax ? v : Tmax);
}

// Blocks of the split kernel that fit the current device at once (SM count x resident blocks per SM).
// Falls back to 148 x 5 (B200, up to 102 registers per thread) when no device can be queried.
template <int D, int G>
int resident_blocks_of() {
  int dev = 0, sms = 0, occ = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 0;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, cowa_decode_split_kernel<D, G>, kThreads, 0) !=
      cudaSuccess)
    return 0;
  return sms * occ;
}

int resident_blocks(int D, int G) {
  static int cache[2][4] = {{0, 0, 0, 0}, {0, 0, 0, 0}};
  const int di = D == 128 ? 1 : 0, gi = G == 1 ? 0 : G == 2 ? 1 : G == 4 ? 2 : 3;
  if (cache[di][gi] == 0) {
    int r = 0;
    if (D == 128) r = G == 1 ? resident_blocks_of<128, 1>() : G == 2 ? resident_blocks_of<128, 2>()
                    : G == 4 ? resident_blocks_of<128, 4>() : resident_blocks_of<128, 8>();
    else r = G == 1 ? resident_blocks_of<64, 1>() : G == 2 ? resident_blocks_of<64, 2>()
             : G == 4 ? resident_blocks_of<64, 4>() : resident_blocks_of<64, 8>();
    if (r <= 0) { cudaGetLastError(); return 148 * 5; }
    cache[di][gi] = r;
  }
  return cache[di][gi];
}

// Splits per (sequence, KV head): the grid should be a whole number of waves of resident
// blocks, each split at most kChunkCap rows (its scores live in shared memory) and not much shorter than
// 128 rows.  `vmax` bounds the visible rows of a block, `units` counts the blocks per split index.
int splits_for(int vmax, int units, int slots) {
  const int by_cap = (vmax + (kChunkCap - 16) - 1) / (kChunkCap - 16);
  const int by_len = (vmax + 127) / 128;
  int s = by_cap;
  for (int waves = 1; waves <= 64; ++waves) {
    s = (int)(((long long)waves * slots) / units);
    if (s >= by_cap && s >= 1) break;
  }
  if (s > by_len) s = by_len;
  if (s < by_cap) s = by_cap;
  return s < 1 ? 1 : s;
}

int pick_splits(int B, int Tmax, int Hq, int Hkv, int D, const cowa_params_t* p) {
  const int hg = p->hkv_global > 0 ? p->hkv_global : Hkv;
  return splits_for(max_visible(Tmax, hg, p), B * Hkv, resident_blocks(D, Hq / Hkv));
}

template <int D>
cudaError_t launch_combine(const DecodeArgs& a, __nv_bfloat16* o, float* lse, cudaStream_t st) {
  const dim3 rows((unsigned)(a.B * a.Hq));
  return a.S > 32 ? cowa::launch_chained(cowa_decode_combine_kernel<D, 16>, rows, 512, 0, st, a, o, lse)
                  : cowa::launch_chained(cowa_decode_combine_kernel<D, 4>, rows, 128, 0, st, a, o, lse);
}

template <int D, int G>
cudaError_t launch_split(const DecodeArgs& a, cudaStream_t st) {
  const dim3 grid(a.S, a.Hkv, a.B);
  return cowa::launch_chained(cowa_decode_split_kernel<D, G>, grid, kThreads, 0, st, a);
}

template <int D>
cudaError_t dispatch_split(int G, const DecodeArgs& a, cudaStream_t st) {
  switch (G) {
    case 1: return launch_split<D, 1>(a, st);
    case 2: return launch_split<D, 2>(a, st);
    case 4: return launch_split<D, 4>(a, st);
    case 8: return launch_split<D, 8>(a, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace

namespace cowa {

int decode_validate(const void* q, const void* kc, const void* vc, const int32_t* lens, const void* o, int B,
                    int Tmax, int Hq, int Hkv, int D, const cowa_params_t* p) {
  if (!q || !kc || !vc || !lens || !o || !p) return COWA_ERR_INVALID_ARG;
  if (B <= 0 || Tmax <= 0 || Hq <= 0 || Hkv <= 0 || Hq % Hkv != 0) return COWA_ERR_INVALID_ARG;
  if (!p->full_attn && (p->sink < 0 || p->local < 1)) return COWA_ERR_INVALID_ARG;
  const int hg = p->hkv_global > 0 ? p->hkv_global : Hkv;
  if (p->hkv_offset < 0 || p->hkv_offset + Hkv > hg) return COWA_ERR_INVALID_ARG;
  if (D != 64 && D != 128) return COWA_ERR_UNSUPPORTED;
  const int G = Hq / Hkv;
  if (G != 1 && G != 2 && G != 4 && G != 8) return COWA_ERR_UNSUPPORTED;
  if (B > 65535 || Hkv > 65535) return COWA_ERR_UNSUPPORTED;
  if (!(p->softmax_scale > 0.f)) return COWA_ERR_INVALID_ARG;
  if (!aligned16(q) || !aligned16(kc) || !aligned16(vc) || !aligned16(o)) return COWA_ERR_MISALIGNED;
  for (int i = 0; i < 3; ++i)
    if (p->q_strides[i] || p->o_strides[i]) return COWA_ERR_UNSUPPORTED;  // q and o of a decode step are [B, Hq, D]
  return COWA_OK;
}

size_t decode_ws_bytes(int B, int Hq, int D, int S) {
  return (size_t)B * Hq * S * (D + 2) * sizeof(float);
}

// Enqueues the split and combine kernels using `ws` (>= decode_ws_bytes) as scratch.
int decode_launch(const void* q, const void* kc, const void* vc, const int32_t* lens, void* o, float* lse,
                  int B, int Tmax, int Hq, int Hkv, int D, const cowa_params_t* p, int S, void* ws,
                  cudaStream_t st) {
  DecodeArgs a;
  a.q = static_cast<const __nv_bfloat16*>(q);
  a.kc = static_cast<const __nv_bfloat16*>(kc);
  a.vc = static_cast<const __nv_bfloat16*>(vc);
  a.lens = lens;
  a.ws_o = static_cast<float*>(ws);
  a.ws_m = a.ws_o + (size_t)B * Hq * S * D;
  a.ws_l = a.ws_m + (size_t)B * Hq * S;
  a.B = B; a.Tmax = Tmax; a.Hq = Hq; a.Hkv = Hkv; a.S = S;
  int rc;
  if ((rc = resolve_strides(p->k_strides, Hkv, Tmax, D, &a.sk))) return rc;
  if ((rc = resolve_strides(p->v_strides, Hkv, Tmax, D, &a.sv))) return rc;
  // No key lies further than Tmax away: wider windows mean the same as Tmax, and sums of widths stay inside 32 bits.
  a.sink = std::min(p->sink, Tmax); a.near = std::min(p->local, Tmax);
  a.hkv_global = p->hkv_global > 0 ? p->hkv_global : Hkv;
  a.hkv_offset = p->hkv_offset;
  a.full_attn = p->full_attn;
  const long long rows = (long long)B * Hkv * max_visible(Tmax, a.hkv_global, p);  // K and V: 4 D bytes each
  a.ahead = rows * D <= (4ll << 20) && rows <= 2ll * kThreads * S * B * Hkv;
  a.scale_log2 = p->softmax_scale * 1.4426950408889634f;
  const int G = Hq / Hkv;
  cudaError_t e = (D == 128) ? dispatch_split<128>(G, a, st) : dispatch_split<64>(G, a, st);
  if (e != cudaSuccess) return record_cuda_error(e);
  e = (D == 128) ? launch_combine<128>(a, static_cast<__nv_bfloat16*>(o), lse, st)
                 : launch_combine<64>(a, static_cast<__nv_bfloat16*>(o), lse, st);
  if (e != cudaSuccess) return record_cuda_error(e);
  return COWA_OK;
}

}  // namespace cowa

extern "C" {

size_t cowa_decode_workspace_bytes(int B, int Tmax, int Hq, int Hkv, int D, const cowa_params_t* p) {
  if (!p || B <= 0 || Tmax <= 0 || Hq <= 0 || Hkv <= 0 || Hq % Hkv != 0 || (D != 64 && D != 128)) return 0;
  return cowa::decode_ws_bytes(B, Hq, D, pick_splits(B, Tmax, Hq, Hkv, D, p));
}

int cowa_decode(const void* q, const void* kcache, const void* vcache, const int32_t* lens, void* o,
                float* lse, int B, int Tmax, int Hq, int Hkv, int D, const cowa_params_t* p,
                void* workspace, size_t workspace_bytes, void* stream) {
  int st = cowa::decode_validate(q, kcache, vcache, lens, o, B, Tmax, Hq, Hkv, D, p);
  if (st != COWA_OK) return st;
  const int S = pick_splits(B, Tmax, Hq, Hkv, D, p);
  if (!workspace) return COWA_ERR_INVALID_ARG;
  if (!cowa::aligned16(workspace)) return COWA_ERR_MISALIGNED;
  if (workspace_bytes < cowa::decode_ws_bytes(B, Hq, D, S)) return COWA_ERR_WORKSPACE_TOO_SMALL;
  return cowa::decode_launch(q, kcache, vcache, lens, o, lse, B, Tmax, Hq, Hkv, D, p, S, workspace,
                             static_cast<cudaStream_t>(stream));
}

size_t cowa_decode_static_capacity(void) { return kStaticScratchBytes; }

int cowa_decode_static(const void* q, const void* kcache, const void* vcache, const int32_t* lens, void* o,
                       float* lse, int B, int Tmax, int Hq, int Hkv, int D, const cowa_params_t* p,
                       void* stream) {
  int st = cowa::decode_validate(q, kcache, vcache, lens, o, B, Tmax, Hq, Hkv, D, p);
  if (st != COWA_OK) return st;
  const int S = pick_splits(B, Tmax, Hq, Hkv, D, p);
  if (cowa::decode_ws_bytes(B, Hq, D, S) > kStaticScratchBytes) return COWA_ERR_STATIC_SCRATCH_EXCEEDED;
  cudaError_t e = cudaSuccess;
  void* scratch = static_scratch_ptr(&e);
  if (!scratch) return cowa::record_cuda_error(e);
  // Every slot of the split states that the merge kernel reads is written by the split kernel of
  // the same call, so nothing left over from an earlier call needs clearing.
  return cowa::decode_launch(q, kcache, vcache, lens, o, lse, B, Tmax, Hq, Hkv, D, p, S, scratch,
                             static_cast<cudaStream_t>(stream));
}

}  // extern "C"
