// Pieces shared by the forward kernels' translation units.
#pragma once
#include <cuda_bf16.h>

#include "cowa_common.h"
#include "cowa_ptx.cuh"
#include "cowa_tma.h"

struct FwdArgs {
  float* lse;
  unsigned int* status;
  int B, Nq, Nk, Hq, Hkv, G;  // packed batches: Nq, Nk unused
  float scale_log2;
  CowaHeadWindows wins;
  // packed (variable-length) batches only
  const int* cu_q;   // [B+1] row offsets of the sequences in q / o / lse
  const int* cu_k;   // [B+1] row offsets in k / v
  __nv_bfloat16* o;  // raw output pointer for the last, partial tile of a sequence
  int total_q, total_k;
  CowaStrides so;    // of o (batched calls)
  int sink, local, hkv_global, hkv_offset, full_attn, explicit_windows;
  int longest_first;  // sequences in order of their keys (varlen_locate_longest), else in the batch's
};

namespace cowa {
// Clusters of two blocks of the pair kernel that the current device holds at once: a block takes an SM, and a cluster lies
// within one GPC, so that some SMs may be left out (74 on the B200 measured).
int resident_pairs();

// Pair kernel (cowa_fwd_pair.cu; the tensor maps of the one-head kernel, 64-row boxes of K and V): two QO heads of a
// group at a time, `items` = tiles x pairs of heads.  split = 1: a block per SM at a time, with `rounds` items for its share
// and others taken over after them; split = 2: every item shared by a cluster of two blocks.
template <int D, bool VARLEN>
int launch_fwd_pair(const CUtensorMap& mq, const CUtensorMap& mk, const CUtensorMap& mv, const CUtensorMap& mo,
                    const FwdArgs& a, long long items, int rounds, int split, cudaStream_t st);
}  // namespace cowa
