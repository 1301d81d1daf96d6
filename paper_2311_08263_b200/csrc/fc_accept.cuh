// Verification, commit, shift and refill of one sequence's window by one warp (all integer work; c <= 64).
#pragma once
#include "fc_internal.h"

namespace fc {

// a[j] = greedy token after window slot j.  a[0] is always exact; a[j] is exact while every guess w[1..j] matched the
// exact token before it (Eq. 5).  K/V of the accepted rows already sit at their final slots, so the commit is kv_len += k.
// New window: pending token a[k-1], the unverified outputs a[k..c-1] as next guesses, then refill ids for the k-1 positions
// no forward has predicted yet.  A lane holds slots lane and lane + 32.
__device__ __forceinline__ void accept_warp(const AcceptArgs &a, int bl, int lane) {
  const int b = a.seq_map ? a.seq_map[bl] : a.b0 + bl, c = a.c;
  int32_t *w = a.window + (long long)b * c;
  if (a.err_inject && bl == 0 && lane == 0) atomicExch(a.err_inject, 1u);
  int arg[2], win[2];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int j = lane + 32 * h, r = bl * c + j;
    arg[h] = win[h] = 0;
    if (j >= c) continue;
    win[h] = w[j];
    if (a.amax) {
      arg[h] = (int32_t)(0xFFFFFFFFu - (unsigned int)(__ldcg(a.amax + r) & 0xFFFFFFFFull));
      if (a.amax_clear) a.amax_clear[r] = 0ull;
    } else {
      arg[h] = a.argmax[r];
    }
  }
  if (a.host_err && bl == 0 && lane == 0) *a.host_err = a.err ? (int32_t)*(volatile const unsigned int *)a.err : 0;
  if (a.done && a.done[b]) {
    if (lane == 0) { a.accepted_count[b] = 0; if (a.host_count) a.host_count[b] = 0; }
    return;
  }
  // guess j is right when it equals the greedy token after slot j - 1
  const int prev0 = __shfl_up_sync(0xffffffffu, arg[0], 1), up1 = __shfl_up_sync(0xffffffffu, arg[1], 1);
  const int last0 = __shfl_sync(0xffffffffu, arg[0], 31), prev1 = lane == 0 ? last0 : up1;
  const bool ok0 = lane == 0 || (lane < c && win[0] == prev0), ok1 = lane + 32 < c && win[1] == prev1;
  const unsigned long long good = (unsigned long long)__ballot_sync(0xffffffffu, ok0) | ((unsigned long long)__ballot_sync(0xffffffffu, ok1) << 32);
  int k = ~good ? __ffsll((long long)~good) - 1 : 64;              // slots 0 .. k-1 are right
  if (k > c) k = c;
  // stop rules: cut at max_tokens and just after the first EOS
  const unsigned long long eos = a.eos_id < 0 ? 0ull :
      (unsigned long long)__ballot_sync(0xffffffffu, lane < c && arg[0] == a.eos_id) | ((unsigned long long)__ballot_sync(0xffffffffu, lane + 32 < c && arg[1] == a.eos_id) << 32);
  const int n0 = a.n_gen[b];
  int kept = k;
  if (a.max_tokens > 0) kept = min(kept, max(0, a.max_tokens - n0));
  const int first_eos = eos ? __ffsll((long long)eos) - 1 : 64;
  bool finished = false;
  if (first_eos < kept) { kept = first_eos + 1; finished = true; }
  if (a.max_tokens > 0 && n0 + kept >= a.max_tokens) finished = true;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int j = lane + 32 * h;
    if (j >= kept) continue;
    a.accepted_tokens[(long long)b * c + j] = arg[h];
    if (a.host_tokens) a.host_tokens[(long long)b * c + j] = arg[h];
    if (a.out_tokens && n0 + j < a.out_stride) a.out_tokens[(long long)b * a.out_stride + n0 + j] = arg[h];
  }
  if (lane == 0) {
    a.accepted_count[b] = kept;
    if (a.host_count) a.host_count[b] = kept;
  }
  if (!a.commit) return;
  __syncwarp();
  if (finished && a.done && lane == 0) a.done[b] = 1;
  k = kept;                                                        // after a cut the remaining state is only reported, never used
  if (k > 0) {
    const int n1 = n0 + k;
    if (lane == 0) { a.kv_len[b] += k; a.n_gen[b] = n1; }
    const int P = a.prompt_lens ? a.prompt_lens[b] : 1;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int j = lane + 32 * h;
      // slot j <- a[k - 1 + j] where there is one
      const int src = k - 1 + j;
      const int s0 = __shfl_sync(0xffffffffu, arg[0], src & 31), s1 = __shfl_sync(0xffffffffu, arg[1], src & 31);
      if (j >= c) continue;
      if (j <= c - k) win[h] = src < 32 ? s0 : s1;
      else win[h] = (a.refill == FC_REFILL_PAD || !a.prompt) ? a.pad_id : a.prompt[(long long)b * a.p_stride + (n1 + j - 1) % P];
      w[j] = win[h];
    }
  }
  if (a.host_window)
#pragma unroll
    for (int h = 0; h < 2; ++h)
      if (lane + 32 * h < c) a.host_window[(long long)b * c + lane + 32 * h] = win[h];
}

}  // namespace fc
