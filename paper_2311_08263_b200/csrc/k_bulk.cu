// Many rows per forward (prompts, large batches): every projection as one dense GEMM of its own, y[R, N] = x[R, K] . W[N, K]^T
// with the activations as a bf16 pair high + low, plus the kernel that makes such a pair.
//
// What bounds it: at a few hundred rows the tensor rate (both halves of the pair are multiplied: 4 R N K flops), then the
// operand bytes out of L2.  So the tile is as large as tensor memory allows with two accumulators: a cluster of two CTAs
// (tcgen05 cta_group::2, M = 256) multiplies 256 weight rows by up to 256 activation rows, and the high and the low products
// go to the SAME accumulator - per k-block of 64 a CTA loads 16 KB of weights once for both halves (48 KB per 2 x 256 x 256 x
// 64 products of the pair; the chained kernel's pairs load 32 KB for half as many).  Gate and up run together: a CTA's 128
// weight rows are 64 of the gate and the same 64 of up, so the two factors of SwiGLU lie 64 lanes apart in one accumulator; the
// two epilogue warps that hold them swap halves of each 16-row block through shared memory and write the down projection's
// operand themselves.  (Two accumulators of 128 rows in the same lanes need no exchange but MMAs of half the width: gate/up of
// 13B at about 1000 rows 444 us that way, 390 this way; a prompt batch of 13B, 8 layers, 63.1 -> 60.1 ms.)
//
// An accumulator in tensor memory runs over six k-blocks only; then the epilogue warps add it to fp32 sums in their
// registers, while the next six run in the other accumulator.  The tensor core's own additions are not rounded to
// nearest, so their number sets the error.  Logits of a 13B step of 256 rows against 64 bits (three seeds), and the time
// of 4 layers: chained launch 1.07 / 1.25 / 1.29e-3; whole k range in one accumulator above 1.5e-3; 8 k-blocks 1.09 / 1.32 /
// 1.28e-3, 1.77 ms; 6: 1.07 / 1.23 / 1.22e-3, 1.82 ms; 4: 1.03 / 1.20 / 1.06e-3, 1.88 ms.
//
// Steps that store very many keys and values (BulkArgs::split) add up as the chained launch does: a high and a low accumulator over
// that launch's chunks of 16 k-blocks, shares cut between chunks.  Their results differ from that launch's by the order of fp32
// additions only.  With other sums the tensor core's rounding differs, which moves more stored K/V values over a bf16 rounding
// boundary (7.0e-4 of layer 0's instead of 3.4e-5), and one such value moves its row of logits by up to a few per cent.  Largest
// difference of two steps of 7B from the chained launch, 512 rows, 24 seeds, in units of the logits' rms: six-block sums 0.0259
// (median 0.0087), split 0.0169 (0.0038), two runs of the chained launch 0.0152 (0.0022); the distance from 64 bits is the same for
// all three.  The accumulators cannot alternate then: the high one is added up while the last low products run, and the next
// chunk waits for the rest (these two steps: six-block sums 30.7 ms, split 31.8, chained launch 35.1).
//
// The tiles of a projection seldom are a whole number of rounds over the pairs: whole rounds run tile by tile, the tiles
// that are left over are dealt as one run of k-blocks, cut into equal shares for all pairs (a share ends in one tile and may
// begin the next).  The pieces of a tile meet in L2: on the residual as fp32 reductions; elsewhere each piece is
// stored and the warp that stores the last one of its part of the tile adds them up, in the order of the pieces, and runs the
// epilogue.  Nobody waits for anybody.
//
// Warps: 0 TMA producer, 1 MMA issuer (the pair's leader issues for both) and tensor-memory owner, 2-9 epilogue.  Persistent:
// pair i takes tiles i, i + pairs, ...; the epilogue of one tile overlaps the MMAs of the next.  Every wait is bounded.
#include <cstring>

#include "fc_internal.h"
#include "fc_ptx.cuh"

namespace fc {

namespace {
constexpr int kBulkThreads = 320;
constexpr int kEpiWarps = 8;
constexpr int kSwapBytes = 16 * 1024;              // BULK_SWIGLU: four pairs of epilogue warps x two buffers x two directions x 1 KB
constexpr int kMaxStages = 8;
constexpr int kWTile = kTileM * kTileK * 2;        // 16 KB: this CTA's 128 weight rows of a k-block
constexpr int kAccKb = 6;                          // k-blocks an accumulator runs over before it is added up in registers
constexpr int kSplitKb = 16;                       // the same with a high and a low accumulator: the chunks of the chained launch
constexpr int kSlotF4 = 1024;                      // one warp's part of a piece: 16 KB
constexpr size_t kBulkSmem = 225 * 1024;           // ring + alignment; static shared memory takes the rest of 227 KB

struct BulkMaps {
  CUtensorMap w[kMaxMats];
  CUtensorMap x;                  // activation pair [2 * pan_rows, K], boxes of 64 k x bn / 2 rows
};

struct BulkParams {
  int n_tiles[kMaxMats], n_mats;  // 256-row weight tiles per matrix
  int y_off[kMaxMats];
  int nkb;                        // 64-wide k-blocks
  int cut_kb;                     // length of a tile in the run that is cut into shares (split: rounded up to whole chunks)
  int n_rt, bn;                   // row tiles, rows per tile
  int n_units;                    // weight tiles x row tiles
  int rounds;                     // rounds of whole units (the last may be partial)
  int share;                      // k-blocks per pair of the units behind them (0: none are left)
  float4 *slots;                  // pieces: [pair][2][rank][epilogue warp][kSlotF4]
  unsigned int *arrived;          // [unit of the last part][rank][epilogue warp], zero outside of a launch
  int stages, stage_bytes;
  int R, pan_rows;
  float *y; int ldy;
  const float *ss; float eps; int dn;           // sums of squares of the normalised input rows (BULK_SWIGLU, BULK_HEAD)
  __nv_bfloat16 *out_pan; int out_rows, out_ld; // BULK_SWIGLU: pair [2][out_rows][out_ld]
  const int32_t *tokens, *perm; float beta;     // BULK_HEAD
  unsigned long long *amax; float *logits; int vocab;
  unsigned int *err;
};

// Two warps (64 threads) meet at named barrier `id`; the verdict is true where it is for every lane of both.
__device__ __forceinline__ bool meet_and(int id, bool ok) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.u32 q, %1, 0;\n\t"
      "bar.red.and.pred p, %2, 64, q;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(r) : "r"((uint32_t)ok), "r"(id) : "memory");
  return r != 0;
}
__device__ __forceinline__ void meet(int id) {
  __syncwarp();
  asm volatile("bar.sync %0, 64;" ::"r"(id) : "memory");
}
__device__ __forceinline__ uint32_t pack_pair(float a, float b) {
  __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<uint32_t *>(&v);
}
__device__ __forceinline__ float lo_of(uint32_t p) { return __uint_as_float(p << 16); }
__device__ __forceinline__ float hi_of(uint32_t p) { return __uint_as_float(p & 0xFFFF0000u); }
}  // namespace

// ------------------------------------------------------------------------------------ activations -> bf16 pair
// One block per row: x * gain as high + low, sum x^2 (the 1/rms factor is applied by the consumer of the product).
__global__ void __launch_bounds__(256) norm_pair_kernel(const float *x, const __nv_bfloat16 *gain, float *ss, __nv_bfloat16 *pan,
                                                         int d, long long lo_off) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  __shared__ float part[8];
  const int r = blockIdx.x;
  const float *px = x + (long long)r * d;
  __nv_bfloat16 *ph = pan + (long long)r * d;
  float sq = 0.f;
  asm volatile("griddepcontrol.wait;" ::: "memory");
  for (int k = threadIdx.x * 8; k < d; k += 256 * 8) {
    const float4 a = __ldcg(reinterpret_cast<const float4 *>(px + k)), b = __ldcg(reinterpret_cast<const float4 *>(px + k + 4));
    const uint4 gq = __ldg(reinterpret_cast<const uint4 *>(gain + k));
    float v[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
    const uint32_t gw[4] = {gq.x, gq.y, gq.z, gq.w};
    uint32_t h[4], l[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      sq = fmaf(v[2 * i], v[2 * i], sq); sq = fmaf(v[2 * i + 1], v[2 * i + 1], sq);
      v[2 * i] *= lo_of(gw[i]); v[2 * i + 1] *= hi_of(gw[i]);
      h[i] = pack_pair(v[2 * i], v[2 * i + 1]);
      l[i] = pack_pair(v[2 * i] - lo_of(h[i]), v[2 * i + 1] - hi_of(h[i]));
    }
    *reinterpret_cast<uint4 *>(ph + k) = make_uint4(h[0], h[1], h[2], h[3]);
    *reinterpret_cast<uint4 *>(ph + lo_off + k) = make_uint4(l[0], l[1], l[2], l[3]);
  }
  sq = warp_sum_f(sq);
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = sq;
  __syncthreads();
  if (threadIdx.x == 0) {
    float t = 0.f;
#pragma unroll
    for (int i = 0; i < 8; ++i) t += part[i];
    ss[r] = t;
  }
}

// ------------------------------------------------------------------------------------ GEMM
template <int EPI, bool SPLIT>
__global__ void __launch_bounds__(kBulkThreads, 1) bulk_gemm_kernel(const __grid_constant__ BulkMaps maps, const __grid_constant__ BulkParams p) {
  constexpr bool kMixed = EPI == BULK_SWIGLU;                     // a CTA's weight rows: 64 of gate, 64 of up
  extern __shared__ unsigned char smem_dyn[];
  __shared__ __align__(8) unsigned long long full_b[kMaxStages], empty_b[kMaxStages], accum_full[2], tmem_empty[2], drain_bar;
  __shared__ uint32_t tmem_base_s;
  __shared__ int abort_s;
  __shared__ unsigned int last_s[4];                              // per pair of epilogue warps: pieces of the tile that were there
  const uint32_t base = (smem_u32(smem_dyn) + 1023u) & ~1023u;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int S = p.stages;
  const uint32_t rank = cluster_rank();                           // 0: the pair's leader
  const int pair = blockIdx.x >> 1, n_pairs = gridDim.x >> 1;
  volatile int *abort_flag = &abort_s;

  if (threadIdx.x == 0) {
    abort_s = 0;
    for (int i = 0; i < kMaxStages; ++i) { mbar_init(smem_u32(&full_b[i]), 1); mbar_init(smem_u32(&empty_b[i]), 1); }
    for (int i = 0; i < 2; ++i) { mbar_init(smem_u32(&accum_full[i]), 1); mbar_init(smem_u32(&tmem_empty[i]), 2 * kEpiWarps); }
    mbar_init(smem_u32(&drain_bar), 1);
    fence_barrier_init();
  }
  if (warp == 1) tmem_alloc_pair(smem_u32(&tmem_base_s), 512);
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();                                             // the peer's barriers exist before anything arrives on them
  tc_fence_after();
  const uint32_t tmem_base = tmem_base_s;
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

  // Item n of this pair: unit u = (weight tile, row tile), k-blocks [kb0, kb1).  Row tiles vary fastest, so that the pairs
  // that run at the same time share weight tiles.
  struct Item { int u, m, lt, rt, kb0, kb1; };
  auto item = [&](int n, Item &t) -> bool {
    if (n < p.rounds) {
      t.u = pair + n * n_pairs;
      if (t.u >= p.n_units) return false;
      t.kb0 = 0; t.kb1 = p.nkb;
    } else {
      const int g0 = pair * p.share, g1 = min(g0 + p.share, (p.n_units - p.rounds * n_pairs) * p.cut_kb);
      const int tile = g0 / p.cut_kb + (n - p.rounds);
      t.kb0 = max(0, g0 - tile * p.cut_kb);
      t.kb1 = min(p.nkb, g1 - tile * p.cut_kb);
      if (p.share == 0 || t.kb0 >= t.kb1) return false;
      t.u = p.rounds * n_pairs + tile;
    }
    t.rt = t.u % p.n_rt;
    t.lt = t.u / p.n_rt;
    t.m = 0;
    if (!kMixed)
      while (t.m + 1 < p.n_mats && t.lt >= p.n_tiles[t.m]) { t.lt -= p.n_tiles[t.m]; ++t.m; }
    return true;
  };
  // Accumulations [kc, acc_end) of an item.  Use u of an accumulator is in buffer u & 1; split: 2 n and 2 n + 1 run side by side.
  auto acc_end = [&](int kc, int kb1) { return min(SPLIT ? (kc / kSplitKb + 1) * kSplitKb : kc + kAccKb, kb1); };
  const uint32_t x_bytes = (uint32_t)p.bn * 64u;                  // one half (high or low) of this CTA's bn / 2 activation rows
  int issued = 0;

  if (warp == 0) {
    if (lane == 0) {
      bool ok = true;
      int it = 0;
      const uint32_t tx = 2u * (uint32_t)(kWTile + 2 * x_bytes);        // both CTAs' bytes count on the leader's barrier
      auto load_w = [&](int stage, int m, int lt, int kb) {
        const uint32_t bar = map_to_cta(smem_u32(&full_b[stage]), 0), dst = base + (uint32_t)(stage * p.stage_bytes);
        if (rank == 0) mbar_expect_tx(smem_u32(&full_b[stage]), tx);
        if (kMixed) {
          const int row = lt * kTileM + (int)rank * (kTileM / 2);
          tma_load_2d_pair(dst, &maps.w[0], kb * kTileK, row, bar);
          tma_load_2d_pair(dst + kWTile / 2, &maps.w[1], kb * kTileK, row, bar);
        } else {
          tma_load_2d_pair(dst, &maps.w[m], kb * kTileK, lt * 2 * kTileM + (int)rank * kTileM, bar);
        }
      };
      auto load_x = [&](int stage, int rt, int kb) {
        const uint32_t bar = map_to_cta(smem_u32(&full_b[stage]), 0), dst = base + (uint32_t)(stage * p.stage_bytes + kWTile);
        const int row = rt * p.bn + (int)rank * (p.bn >> 1);
        tma_load_2d_pair(dst, &maps.x, kb * kTileK, row, bar);
        tma_load_2d_pair(dst + x_bytes, &maps.x, kb * kTileK, p.pan_rows + row, bar);
      };
      bool first = true;
      Item t;
      for (int n = 0; ok && item(n, t); ++n) {
        int kb = t.kb0;
        if (first) {
          // weights depend on nothing that runs on the device: the ring's first round of them is requested before the
          // kernel in front has finished, the activations after
          const int pre = min(S, t.kb1 - t.kb0);
          for (int i = 0; i < pre; ++i) load_w(i, t.m, t.lt, t.kb0 + i);
          asm volatile("griddepcontrol.wait;" ::: "memory");
          asm volatile("fence.proxy.async;" ::: "memory");        // activations stored by the kernel in front, read by the TMA
          for (int i = 0; i < pre; ++i) load_x(i, t.rt, t.kb0 + i);
          kb += pre; it = pre; issued = pre;
          first = false;
        }
        for (; kb < t.kb1; ++kb, ++it) {
          const int stage = it % S;
          if (it >= S && !mbar_wait(smem_u32(&empty_b[stage]), (uint32_t)(it / S - 1) & 1u, abort_flag)) { ok = false; break; }
          load_w(stage, t.m, t.lt, kb);
          load_x(stage, t.rt, kb);
          issued = it + 1;
        }
      }
      // the leader's MMA completions arrive on this CTA's ring barriers too: all of them have landed before it leaves
      for (int i = (it > S ? it - S : 0); i < it && ok; ++i)
        ok = mbar_wait(smem_u32(&empty_b[i % S]), (uint32_t)(i / S) & 1u, abort_flag);
    }
  } else if (warp == 1) {
    if (lane == 0 && rank == 0) {
      bool ok = true;
      int it = 0, uses = 0;
      auto drained = [&](int u) {                                  // buffer u & 1 has been added up since its last use
        if (u >= 2 && !mbar_wait(smem_u32(&tmem_empty[u & 1]), ((uint32_t)(u >> 1) - 1u) & 1u, abort_flag)) return false;
        tc_fence_after();
        return true;
      };
      const uint32_t idesc = make_idesc(p.bn, 2 * kTileM);
      Item t;
      for (int n = 0; ok && item(n, t); ++n)
        for (int kc = t.kb0, kc1; kc < t.kb1 && ok; kc = kc1, uses += SPLIT ? 2 : 1) {
          kc1 = acc_end(kc, t.kb1);
          if (!drained(uses)) { ok = false; break; }
          const uint32_t d0 = tmem_base + (uint32_t)((uses & 1) * 256);
          for (int kb = kc; kb < kc1; ++kb, ++it) {
            const int stage = it % S;
            if (!mbar_wait(smem_u32(&full_b[stage]), (uint32_t)(it / S) & 1u, abort_flag)) { ok = false; break; }
            tc_fence_after();
            const uint32_t sb = base + (uint32_t)(stage * p.stage_bytes);
            const uint64_t a0 = smem_desc_sw128(sb);
            const uint64_t bh = smem_desc_sw128(sb + kWTile), bl = smem_desc_sw128(sb + kWTile + x_bytes);
            if constexpr (SPLIT) {
#pragma unroll
              for (int kk = 0; kk < kTileK / 16; ++kk)
                umma_bf16_pair(d0, a0 + (uint64_t)(kk * 2), bh + (uint64_t)(kk * 2), idesc, (kb > kc || kk > 0) ? 1u : 0u);
              if (kb + 1 == kc1) umma_commit_pair(smem_u32(&accum_full[0]));
              if (kb == kc && !drained(uses + 1)) { ok = false; break; }
#pragma unroll
              for (int kk = 0; kk < kTileK / 16; ++kk)
                umma_bf16_pair(d0 + 256, a0 + (uint64_t)(kk * 2), bl + (uint64_t)(kk * 2), idesc, (kb > kc || kk > 0) ? 1u : 0u);
            } else {
#pragma unroll
              for (int kk = 0; kk < kTileK / 16; ++kk) {
                const uint64_t o = (uint64_t)(kk * 2);
                const uint32_t more = (kb > kc || kk > 0) ? 1u : 0u;
                umma_bf16_pair(d0, a0 + o, bh + o, idesc, more);
                umma_bf16_pair(d0, a0 + o, bl + o, idesc, 1u);
              }
            }
            umma_commit_pair(smem_u32(&empty_b[stage]));
          }
          if (ok) umma_commit_pair(smem_u32(&accum_full[(uses + SPLIT) & 1]));
        }
      // the peer's epilogue warps arrive on this CTA's accumulator barriers: wait for the last two uses
      for (int u = (uses > 2 ? uses - 2 : 0); u < uses && ok; ++u)
        ok = mbar_wait(smem_u32(&tmem_empty[u & 1]), ((uint32_t)u >> 1) & 1u, abort_flag);
    }
  } else {
    asm volatile("griddepcontrol.wait;" ::: "memory");            // outputs may still be read by the kernel in front
    const int q = warp & 3, half = (warp - 2) >> 2;               // tensor-memory lanes 32 q .. 32 q + 31; every second block of 16 rows
    const uint32_t t_lane = tmem_base + ((uint32_t)(q * 32) << 16);
    constexpr int kBlocks = 8;                                    // blocks of 16 rows of a tile that this warp holds
    float sum[kBlocks][16];
    const int duo = half * 2 + (q & 1);                            // BULK_SWIGLU: the two warps of the same columns
    const bool is_up = q >= 2;
    float *swap = reinterpret_cast<float *>(smem_dyn + (base - smem_u32(smem_dyn)) + (size_t)S * p.stage_bytes) + duo * 1024;
    Item t;
    int use = 0;
    bool ok = true;
    for (int n = 0; item(n, t); ++n) {
      const int m = t.m;
      const int r_base = t.rt * p.bn + half * 16;                  // first row of block 0
      const int blocks = min((p.bn - half * 16 + 31) >> 5, (p.R - r_base + 31) >> 5);      // blocks with rows in them
      for (int kc = t.kb0, low = 0; kc < t.kb1; ++use) {
        const int acc = use & 1;
        ok = mbar_wait_warp(smem_u32(&accum_full[acc]), ((uint32_t)use >> 1) & 1u, abort_flag);
        if (kMixed) ok = meet_and(1 + duo, ok);                    // both go on or both leave
        if (!ok) break;
        tc_fence_after();
        const uint32_t t_acc = t_lane + (uint32_t)(acc * 256 + half * 16);
        const bool more = kc > t.kb0 || low;
#pragma unroll
        for (int i = 0; i < kBlocks; ++i) {
          if (i < blocks) {
            float v[16];
            tmem_ld16(t_acc + (uint32_t)(i * 32), v);
#pragma unroll
            for (int j = 0; j < 16; ++j) sum[i][j] = more ? sum[i][j] + v[j] : v[j];
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(map_to_cta(smem_u32(&tmem_empty[acc]), 0));
        if (SPLIT && !low) low = 1;                              // the low products of the same chunk
        else { kc = acc_end(kc, t.kb1); low = 0; }
      }
      if (!ok) break;
      if (EPI != BULK_ADD && (t.kb0 > 0 || t.kb1 < p.nkb)) {       // a piece of a tile
        const int tile = t.u - p.rounds * n_pairs;
        const int from = tile * p.cut_kb / p.share, to = ((tile + 1) * p.cut_kb - 1) / p.share;      // the pairs that hold its pieces
        auto slot_of = [&](int pr) -> float4 * {
          const int second = pr * p.share / p.cut_kb != tile;
          return p.slots + ((size_t)((pr * 2 + second) * 2 + (int)rank) * kEpiWarps + (warp - 2)) * kSlotF4 + lane;
        };
        float4 *dst = slot_of(pair);
#pragma unroll
        for (int i = 0; i < kBlocks; ++i)
          if (i < blocks)
#pragma unroll
            for (int k4 = 0; k4 < 4; ++k4)
              __stcg(dst + (i * 4 + k4) * 32, make_float4(sum[i][4 * k4], sum[i][4 * k4 + 1], sum[i][4 * k4 + 2], sum[i][4 * k4 + 3]));
        __threadfence();                                           // this lane's piece is visible before the count
        __syncwarp();
        if (kMixed) meet(1 + duo);                                 // the two warps of a column count as one
        unsigned int before = 0;
        if (lane == 0 && !(kMixed && is_up)) {
          unsigned int *word = p.arrived + ((size_t)tile * 2 + rank) * kEpiWarps + (kMixed ? duo : warp - 2);
          __threadfence();
          before = atomicAdd(word, 1u);
          if (before == (unsigned int)(to - from)) *word = 0u;     // the last one: nobody else touches it in this launch
          if (kMixed) last_s[duo] = before;
        }
        if (kMixed) {
          meet(1 + duo);
          before = last_s[duo];
        } else {
          before = __shfl_sync(0xffffffffu, before, 0);
        }
        if (before != (unsigned int)(to - from)) continue;
        __threadfence();
        for (int pr = from; pr <= to; ++pr) {
          const float4 *src = slot_of(pr);
#pragma unroll
          for (int i = 0; i < kBlocks; ++i)
            if (i < blocks)
#pragma unroll
              for (int k4 = 0; k4 < 4; ++k4) {
                const float4 x = __ldcg(src + (i * 4 + k4) * 32);
                float *sd = &sum[i][4 * k4];
                if (pr == from) { sd[0] = x.x; sd[1] = x.y; sd[2] = x.z; sd[3] = x.w; }
                else { sd[0] += x.x; sd[1] += x.y; sd[2] += x.z; sd[3] += x.w; }
              }
        }
      }
      // a lane holds output column n0 + lane for 16 rows of a block; quads are transposed, so that a lane then holds four
      // adjacent columns of rows (lane & 3) + 4 i
      const int n0 = kMixed ? t.lt * kTileM + (int)rank * (kTileM / 2) + (q & 1) * 32 : t.lt * 2 * kTileM + (int)rank * kTileM + q * 32;
#pragma unroll
      for (int i = 0; i < kBlocks; ++i) {
        if (i >= blocks) break;
        const int r0 = r_base + i * 32;
        float (&v)[16] = sum[i];
        if constexpr (EPI == BULK_STORE || EPI == BULK_ADD) {
          float *yb = p.y + p.y_off[m] + n0 + (lane & ~3);
#pragma unroll
          for (int k4 = 0; k4 < 4; ++k4) {
            quad_transpose(v[4 * k4], v[4 * k4 + 1], v[4 * k4 + 2], v[4 * k4 + 3], lane);
            const int r = r0 + 4 * k4 + (lane & 3);
            if (r < p.R) {
              float *dst = yb + (long long)r * p.ldy;
              if (EPI == BULK_STORE) *reinterpret_cast<float4 *>(dst) = make_float4(v[4 * k4], v[4 * k4 + 1], v[4 * k4 + 2], v[4 * k4 + 3]);
              else red_add_v4(dst, v[4 * k4], v[4 * k4 + 1], v[4 * k4 + 2], v[4 * k4 + 3]);
            }
          }
        } else if constexpr (EPI == BULK_SWIGLU) {
          // the gate warp keeps rows 0-7 of the block and gets their up factors, the up warp rows 8-15 and their gates
          float *out = swap + (i & 1) * 512 + (is_up ? 256 : 0) + lane, *in = swap + (i & 1) * 512 + (is_up ? 0 : 256) + lane;
#pragma unroll
          for (int j = 0; j < 8; ++j) out[j * 32] = is_up ? v[j] : v[8 + j];
          const int ra = r0 + (is_up ? 8 : 0), rs = ra + (lane & 7);
          const float s_mine = rs < p.R ? rsqrtf(__ldcg(p.ss + rs) / (float)p.dn + p.eps) : 0.f;
          meet(1 + duo);                                           // (two buffers in turn: a block's reader is past it one barrier later)
          float y[8];
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const float other = in[j * 32], own = is_up ? v[8 + j] : v[j];
            const float s = __shfl_sync(0xffffffffu, s_mine, j);
            const float gt = s * (is_up ? other : own);
            y[j] = __fdividef(gt, 1.0f + __expf(-gt)) * (s * (is_up ? own : other));
          }
#pragma unroll
          for (int k4 = 0; k4 < 2; ++k4) {
            quad_transpose(y[4 * k4], y[4 * k4 + 1], y[4 * k4 + 2], y[4 * k4 + 3], lane);
            const int r = ra + 4 * k4 + (lane & 3);
            if (r < p.R) {
              const uint32_t h0 = pack_pair(y[4 * k4], y[4 * k4 + 1]), h1 = pack_pair(y[4 * k4 + 2], y[4 * k4 + 3]);
              __nv_bfloat16 *dst = p.out_pan + (long long)r * p.out_ld + n0 + (lane & ~3);
              *reinterpret_cast<uint2 *>(dst) = make_uint2(h0, h1);
              *reinterpret_cast<uint2 *>(dst + (long long)p.out_rows * p.out_ld) =
                  make_uint2(pack_pair(y[4 * k4] - lo_of(h0), y[4 * k4 + 1] - hi_of(h0)), pack_pair(y[4 * k4 + 2] - lo_of(h1), y[4 * k4 + 3] - hi_of(h1)));
            }
          }
        } else {                                                  // BULK_HEAD: logits, bias, running maximum per row
          const int col = n0 + lane;
          const int rs = r0 + (lane & 15);
          const float s_mine = rs < p.R ? rsqrtf(__ldcg(p.ss + rs) / (float)p.dn + p.eps) : 0.f;
          const int f_mine = p.perm && rs < p.R ? p.perm[p.tokens[rs]] : -1;
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            const int r = r0 + j;
            const float s = __shfl_sync(0xffffffffu, s_mine, j);
            const int f = __shfl_sync(0xffffffffu, f_mine, j);
            if (r < p.R) {
              float logit = v[j] * s;
              if (f == col) logit += p.beta;
              if (p.logits) p.logits[(long long)r * p.vocab + col] = logit;
              const unsigned long long key = warp_max_u64(((unsigned long long)ordered_key_u(logit) << 32) | (unsigned long long)(0xFFFFFFFFu - (unsigned int)col));
              if (lane == 0) atomicMax(&p.amax[r], key);
            }
          }
        }
      }
    }
  }

  // ---------------------------------------------------------------- teardown
  __syncthreads();
  if (abort_s) {
    if (threadIdx.x == 0) {
      atomicExch(p.err, 1u);
      // wait (bounded) for copies still in flight: a pair's copies are counted by its leader, and the peer stays until the
      // leader has passed the cluster barrier below
      const unsigned long long t0 = clock64();
      for (int i = (issued > S ? issued - S : 0); i < issued && rank == 0; ++i)
        while (!mbar_try(smem_u32(&full_b[i % S]), (uint32_t)(i / S) & 1u))
          if ((unsigned long long)(clock64() - t0) > kSpinBudget / 4) break;
    }
    if (warp == 1 && lane == 0 && rank == 0) {
      umma_commit_pair(smem_u32(&drain_bar));
      const unsigned long long t0 = clock64();
      while (!mbar_try(smem_u32(&drain_bar), 0u))
        if ((unsigned long long)(clock64() - t0) > kSpinBudget / 4) break;
    }
    __syncthreads();
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();                          // neither CTA leaves, or frees tensor memory, while its peer still works
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc_pair(tmem_base, 512);
  }
}

// ------------------------------------------------------------------------------------ host side
cudaError_t launch_norm_pair(const float *x, const void *gain, float *ss, void *pan, int pan_rows, int R, int d, int pdl, cudaStream_t st) {
  if (R < 1 || d % 8) return cudaErrorInvalidValue;
  cudaLaunchConfig_t cfg;
  memset(&cfg, 0, sizeof cfg);
  cfg.gridDim = dim3(R); cfg.blockDim = dim3(256); cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr; cfg.numAttrs = pdl ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, norm_pair_kernel, x, (const __nv_bfloat16 *)gain, ss, (__nv_bfloat16 *)pan, d, (long long)pan_rows * d);
}

// Rows per tile (a multiple of 32: the N step of a two-CTA MMA) and how the units are dealt.  Cost in tensor cycles: a
// k-block takes the slower of its MMAs (4 cycles per row) and its operand loads (about 56 bytes per cycle and
// SM out of L2); whole rounds take nkb of them, the shares of what is left over `share`, and pieces that have to be stored
// and added up about 9000 besides.
// The shares are whole groups of four k-blocks (an accumulation starts where a share does, so they need not be whole
// accumulations); with split accumulators, whole chunks.
static void bulk_plan(int n_wt, int nkb, int R, int n_pairs, bool add, bool may_share, bool split, int &bn, int &rounds, int &share) {
  const int unit = split ? kSplitKb : 4;
  double best = 0;
  for (int b = 64; b <= 256; b += 32) {
    const long long units = (long long)n_wt * ((R + b - 1) / b);
    const double mma = 4.0 * b, load = (16384 + b * 128) / 56.0, kb = mma > load ? mma : load;
    const long long whole = units / n_pairs, left = units - whole * n_pairs;
    double cost = (double)(whole + (left > 0)) * nkb * kb;
    int r = (int)(whole + (left > 0)), s = 0;
    if (left > 0 && may_share) {
      const long long run = left * (split ? (nkb + unit - 1) / unit * unit : nkb);
      const int per = (int)(((run + n_pairs - 1) / n_pairs + unit - 1) / unit * unit);
      const double c = (whole * (double)nkb + per) * kb + (add ? 2000.0 + 4.0 * b : 9000.0);
      if (per < nkb && c < cost) { cost = c; r = (int)whole; s = per; }
    }
    cost += 1500.0 * (r + (s > 0));
    if (best == 0 || cost < best) { best = cost; bn = b; rounds = r; share = s; }
    if (b >= R) break;
  }
}

template <int EPI, bool SPLIT>
static cudaError_t launch_bulk_t(const BulkMaps &maps, const BulkParams &p, int grid, int pdl, cudaStream_t st) {
  static bool attr_done[kMaxDevices] = {false};
  const int dev = current_device_slot();
  if (!attr_done[dev]) {
    cudaError_t e = cudaFuncSetAttribute(bulk_gemm_kernel<EPI, SPLIT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kBulkSmem);
    if (e != cudaSuccess) return e;
    attr_done[dev] = true;
  }
  cudaLaunchConfig_t cfg;
  memset(&cfg, 0, sizeof cfg);
  cfg.gridDim = dim3(grid); cfg.blockDim = dim3(kBulkThreads); cfg.dynamicSmemBytes = kBulkSmem; cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr; cfg.numAttrs = pdl ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, bulk_gemm_kernel<EPI, SPLIT>, maps, p);
}

cudaError_t launch_bulk_gemm(const UmmaPlan *plan, const BulkArgs &a, int epi, int n_sms, int pdl, cudaStream_t st) {
  BulkMaps maps;
  BulkParams p;
  memset(&p, 0, sizeof p);
  int n_rows[kMaxMats], K;
  const void *weights[kMaxMats];
  umma_plan_view(plan, maps.w, weights, n_rows, p.y_off, p.n_mats, K, p.err);
  int n_wt = 0;
  for (int m = 0; m < p.n_mats; ++m) {
    if (n_rows[m] % (2 * kTileM)) return cudaErrorInvalidValue;
    p.n_tiles[m] = n_rows[m] / (2 * kTileM);
    n_wt += p.n_tiles[m];
  }
  const bool mixed = epi == BULK_SWIGLU;
  if (mixed && (p.n_mats != 2 || n_rows[0] != n_rows[1])) return cudaErrorInvalidValue;      // n_wt: tiles of 128 + 128 rows
  if (epi == BULK_HEAD && p.n_mats != 1) return cudaErrorInvalidValue;
  if (a.R < 1 || a.R > a.pan_rows) return cudaErrorInvalidValue;
  const int n_pairs = n_sms / 2;
  p.nkb = (K + kTileK - 1) / kTileK;
  p.cut_kb = a.split ? (p.nkb + kSplitKb - 1) / kSplitKb * kSplitKb : p.nkb;
  const bool add = epi == BULK_ADD;
  bulk_plan(n_wt, p.nkb, a.R, n_pairs, add, add || (a.slots && n_pairs <= kBulkPairs), a.split != 0, p.bn, p.rounds, p.share);
  p.slots = (float4 *)a.slots; p.arrived = a.arrived;
  p.n_rt = (a.R + p.bn - 1) / p.bn;
  const long long units = (long long)n_wt * p.n_rt;
  if (units > 0x3fffffff) return cudaErrorInvalidValue;
  p.n_units = (int)units;
  p.stage_bytes = kWTile + p.bn * 128;
  p.stages = (int)((kBulkSmem - 1024 - (mixed ? kSwapBytes : 0)) / p.stage_bytes);
  if (p.stages > kMaxStages) p.stages = kMaxStages;
  cudaError_t e = make_pair_tensor_map(&maps.x, a.pan, a.pan_rows, K, p.bn / 2);
  // gate and up: boxes of 64 weight rows
  for (int m = 0; m < 2 && mixed && e == cudaSuccess; ++m) e = make_pair_tensor_map(&maps.w[m], weights[m], n_rows[m] / 2, K, kTileM / 2);
  if (e != cudaSuccess) return e;
  p.R = a.R; p.pan_rows = a.pan_rows; p.y = a.y; p.ldy = a.ldy; p.ss = a.ss; p.eps = a.eps; p.dn = a.dn;
  p.out_pan = (__nv_bfloat16 *)a.out_pan; p.out_rows = a.pan_rows; p.out_ld = mixed ? n_rows[0] : 0;
  p.tokens = a.tokens; p.perm = a.perm; p.beta = a.beta; p.amax = a.amax; p.logits = a.logits; p.vocab = n_rows[0];
  // the shares are cut for all pairs; whole units need no more pairs than there are units
  const int grid = 2 * (p.share > 0 || p.n_units > n_pairs ? n_pairs : p.n_units);
  switch (epi) {
    case BULK_STORE: return a.split ? launch_bulk_t<BULK_STORE, true>(maps, p, grid, pdl, st) : launch_bulk_t<BULK_STORE, false>(maps, p, grid, pdl, st);
    case BULK_ADD: return a.split ? launch_bulk_t<BULK_ADD, true>(maps, p, grid, pdl, st) : launch_bulk_t<BULK_ADD, false>(maps, p, grid, pdl, st);
    case BULK_SWIGLU: return a.split ? launch_bulk_t<BULK_SWIGLU, true>(maps, p, grid, pdl, st) : launch_bulk_t<BULK_SWIGLU, false>(maps, p, grid, pdl, st);
    case BULK_HEAD: return a.split ? launch_bulk_t<BULK_HEAD, true>(maps, p, grid, pdl, st) : launch_bulk_t<BULK_HEAD, false>(maps, p, grid, pdl, st);
  }
  return cudaErrorInvalidValue;
}

size_t bulk_slot_bytes() { return (size_t)kBulkPairs * 2 * 2 * kEpiWarps * kSlotF4 * sizeof(float4); }

}  // namespace fc
