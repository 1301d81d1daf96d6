// Projections of up to 64 rows, y[R, N] = x[R, K] . W[N, K]^T, with ONE writer per output: the projections between two
// attention launches (O, gate/up, down, next layer's QKV) run one after the other in one persistent launch.
//
// What bounds it: the weight stream out of HBM, and at every projection's end the latency until its results are the next
// one's operand.  Partial sums that meet in L2 (the chained launch of k_umma.cu) cost reductions, a release per chunk and
// a conversion of fp32 sums by every CTA that reads them.  Here a cluster of four CTAs owns a run of output columns (weight rows,
// in units of 16): each CTA multiplies them by a quarter of the k range, the four partial sums meet in the cluster's shared
// memory (st.async into the CTA that owns a quarter of the columns), and that CTA writes the finished values once - the
// residual, the bf16 high/low operand pair of the next projection (RMSNorm gain or SwiGLU applied) and its share of the
// row sums of squares.  So activations are operands in memory, loaded by TMA, and nothing is converted twice; results do not
// depend on the order in which CTAs arrive.
//
// Per CTA a ring of 32 KB stages: up to 128 weight rows x two k-blocks of 64 in one TMA box.  (One thread that requests and
// one that consumes cost about 0.25 us per stage whatever its size: 132 CTAs, stages of one k-block 5.3 TB/s, of two 6.8, whatever the
// depth; boxes of 16 rows 3.7.)  The weight stream does not wait for anything but free stages, so it runs ahead into
// the next projection while the results of this one are exchanged.
//
// tcgen05.mma, M = 128 weight rows, N = 2 x BN: the high and the low activation rows side by side, fp32 accumulators in
// tensor memory.  An accumulator runs over four k-blocks; then eight warps add it to fp32 sums in their registers (the
// tensor core's own additions are not rounded to nearest).
//
// Gate and up are finished column range by column range; the last range is published on its own, and down takes the k range of the
// others first, so that the exchange between them costs nothing.
//
// Warps: 0 weights, 1 MMA and tensor memory, 2 activations, 3-10 accumulators -> registers -> cluster, 11-14 cluster -> results.
// Every wait is bounded.  The grid barrier between projections needs every cluster resident: the grid is what
// cudaOccupancyMaxActiveClusters reports.
#include <array>
#include <cstdio>
#include <cstring>
#include <new>
#include <vector>

#include "fc_internal.h"
#include "fc_plan.h"
#include "fc_ptx.cuh"

namespace fc {

namespace {
constexpr int kCl = 4;                             // CTAs per cluster = shares of the k range
constexpr int kUnit = 16;                          // weight rows per unit
constexpr int kTileUnits = 8;                      // units per tile at most (M = 128)
constexpr int kFewestClusters = 16;                // a B200 holds 33
constexpr int kThreadsCl = 480;
constexpr int kDrainWarp0 = 3, kOutWarp0 = 11;
constexpr int kStageW = 2 * kTileM * kTileK * 2;   // 32 KB: two k-blocks
constexpr int kXRow = 16;                          // floats per weight row in an exchange buffer
constexpr int kXBuf = kCl * 32 * kXRow * 4;        // one exchange unit: 32 weight rows x 16 rows from four CTAs
constexpr size_t kMaxSmem = 227 * 1024 - 3 * 1024; // dynamic: the static part takes less than 3 KB
enum { PH_QKV = 0, PH_O = 1, PH_GU = 2, PH_DOWN = 3, PH_HEAD = 4 };
constexpr int kMats = 7;                           // wq (or the LM head), wk, wv, wo, gate, up, down: the matrices of a launch

template <int BN>
struct ClCfg {
  // Tiles whose sums a warp holds at a time: gate and up of a column range.  (Four, activations loaded half as often: 7B, 16 rows
  // 2814 us a step against 2796, 2 x 16 rows 3105 against 3059 - the drain loop is unrolled over them.)
  static constexpr int T = 2;
  static constexpr int H = BN / 2;                                // rows (accumulator columns) per drain warp
  static constexpr int kAcc = 2 * BN;
  static constexpr int NACC = BN == 64 ? 4 : 8;
  static constexpr uint32_t kCols = (uint32_t)(kAcc * NACC);      // 256, 512, 512
  static constexpr int XK = BN == 64 ? 1 : 2;                     // k-blocks per activation slot
  static constexpr int kXBlock = 2 * BN * 128;                    // a k-block, high and low
  static constexpr int kXSlot = XK * kXBlock;
  // Activation slots.  (16 rows: three 2842 us a step, four 2814, five the same; 64 rows: four 4879, five 4794; 32 rows, nine of one
  // k-block instead of four of two: 3142 against 3105.)
  static constexpr int NX = BN == 64 ? 5 : 4;
  static constexpr int NCB = BN / 16;                             // exchange units per tile
  static constexpr int NXB = NCB > 2 ? NCB : 2;                   // exchange buffers: unit u of a launch takes buffer u modulo NXB, so a
                                                                  // buffer always has the same senders, none of which can fall two uses behind
  static constexpr int S = BN == 64 ? 3 : BN == 32 ? 4 : 5;
  static constexpr size_t kSmem = 1024 + (size_t)S * kStageW + NX * kXSlot + NXB * kXBuf;
  static_assert(kSmem <= kMaxSmem, "shared memory");
};

// By value in the launch's parameters, as in all kernels here: a map that lies in global memory would need a proxy fence in every
// block before its first use.  (Other addresses every launch: 7B, 1 row 2606 -> 2632 us a step, 16 rows 2682 -> 2705, 1.1B 923 -> 924; prefetched by
// the set-up warp 2630, 2707, 936.)
struct ClMaps {
  CUtensorMap x[3];                                // operand pairs: residual x gain (K = d), attention (qd), feed-forward (f)
  CUtensorMap w[kMats][2];                         // weights, boxes of the matrix's two tile heights
};

// One kind of projection, as far as it is the same for all clusters (made on the host: integer divisions and their code cost
// every role of every launch).
struct Kind {
  int units, parts, n_tiles;                       // units of the (first) matrix, column ranges, tiles per cluster
  unsigned int inv_parts;                          // reciprocal() of parts
  int early;                                       // gate/up: tiles in front of the last column range (their results are published first)
  int pairs, first;                                // pairs of k-blocks; down: those in front of the last column range of gate/up
  int mat0, h0;                                    // ClMaps::w: first matrix; the lower of the tile heights (the other is one more)
};

struct ClParams {
  Kind kind[5];
  Kind kv;                                         // the K or V matrix of QKV
  unsigned int inv_ncl;                            // reciprocal() of the clusters
  int first, last;                                 // projections [first, last): 4 * layer + PH_*, 4 * n_layers: the LM head
  int n_layers, d, qd, kvd, f, vocab, R;
  float *x, *qkv;
  __nv_bfloat16 *pan_x, *pan_h;                    // [2][kClusterRows][d], [2][kClusterRows][f]
  const __nv_bfloat16 *g_ffn, *g_next;             // gains applied behind O and behind down
  float *ss_x, *ss_ffn, *ss_attn;                  // sums of squares: one slot of kClusterRows per CTA; ss_attn: per row
  int first_slots;                                 // slots of ss_x in front of layer 0
  float eps; int dn;
  unsigned int *bar;                               // two counters per projection (all results, the first column ranges), zero when a forward starts
  unsigned int arrivals;                           // that complete a counter: the CTAs (a test may ask for one more)
  const int32_t *tokens, *perm; float beta;
  unsigned long long *amax; float *logits;
  unsigned int *err;
};

// The units of a matrix are cut into column ranges of nearly equal size, and every range into one tile per cluster: so
// all clusters have the same number of tiles, and with the tiles of one index a whole range of columns is finished.
__host__ __device__ inline void tile_units(const Kind &k, int t, int cl, unsigned int inv_ncl, int &u, int &h) {
  const int b = quotient(t * k.units, k.inv_parts), n = quotient((t + 1) * k.units, k.inv_parts) - b;
  u = b + quotient(cl * n, inv_ncl);
  h = b + quotient((cl + 1) * n, inv_ncl) - u;
}

struct Phase {
  int kind, n_tiles, early, cl;
  int p0, np0, q0, np;                             // this CTA's np pairs of k-blocks: np0 from pair p0, the rest from pair q0
  // tile t: matrix, first unit, height (0 to 8 units; 0: nothing, for a range of fewer units than clusters)
  __device__ __forceinline__ void tile(const ClParams &p, int t, int &mat, int &u, int &h) const {
    const Kind &k = p.kind[kind];
    mat = 0;
    if (kind == PH_GU) {                           // gate and up of the same columns one after the other
      mat = t & 1;
      tile_units(k, t >> 1, cl, p.inv_ncl, u, h);
    } else if (kind == PH_QKV && t >= k.parts) {   // the matrices' taller tiles fall on different clusters
      const int ncl = gridDim.x / kCl;
      mat = t < k.parts + p.kv.parts ? 1 : 2;
      const int c = cl + (mat == 1 ? ncl / 3 : 2 * (ncl / 3));
      tile_units(p.kv, t - k.parts - (mat - 1) * p.kv.parts, c < ncl ? c : c - ncl, p.inv_ncl, u, h);
    } else {
      tile_units(k, t, cl, p.inv_ncl, u, h);
    }
  }
  __device__ __forceinline__ int pair(int i) const { return i < np0 ? p0 + i : q0 + (i - np0); }
  template <int T> __device__ __forceinline__ int pass_end(int t0) const { return min(t0 + T, t0 < early ? early : n_tiles); }
};

__device__ __forceinline__ Phase phase_of(const ClParams &p, int id, int cl, int rank) {
  Phase ph;
  const int l = id >> 2;
  ph.kind = l == p.n_layers ? (int)PH_HEAD : id & 3;
  const Kind &k = p.kind[ph.kind];
  ph.cl = cl; ph.n_tiles = k.n_tiles; ph.early = k.early;
  // down takes its k range in two pieces: the columns that gate/up publishes first, then the rest
  const int rest = k.pairs - k.first;
  ph.p0 = rank * k.first / kCl;
  ph.np0 = (rank + 1) * k.first / kCl - ph.p0;
  ph.q0 = k.first + rank * rest / kCl;
  ph.np = ph.np0 + k.first + (rank + 1) * rest / kCl - ph.q0;
  return ph;
}

__device__ __forceinline__ void load_3d(uint32_t dst, const CUtensorMap *map, int x, int y, int z, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
      ::"r"(dst), "l"(map), "r"(x), "r"(y), "r"(z), "r"(bar) : "memory");
}
__device__ __forceinline__ void load_4d(uint32_t dst, const CUtensorMap *map, int x, int y, int z, int w, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];"
      ::"r"(dst), "l"(map), "r"(x), "r"(y), "r"(z), "r"(w), "r"(bar) : "memory");
}
// Arrival on a barrier of another CTA of the cluster, behind this warp's accesses to its own CTA's shared memory.  (The release is
// restricted to those: an unrestricted one waits for all global stores on their way too, 0.7 us per exchange unit; 8 layers of 1.1B, 16 rows
// 387 us against 350, 64 rows 774 against 594.)
__device__ __forceinline__ void mbar_arrive_far(uint32_t bar_cluster) {
  asm volatile("fence.release.sync_restrict::shared::cta.cluster;" ::: "memory");
  asm volatile("mbarrier.arrive.relaxed.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar_cluster) : "memory");
}
// Bounded wait of a converged warp for what other CTAs of the cluster signal: acquires at cluster scope.
__device__ __forceinline__ bool mbar_try_far(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.b32 %0, 1, 0, p;\n\t}"
      : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
  return ok != 0;
}
__device__ __forceinline__ bool wait_far(uint32_t bar, uint32_t parity, volatile int *abort_flag) {
  bool ok = true;
  if (!mbar_try_far(bar, parity)) {
    const unsigned long long t0 = clock64();
    unsigned int spins = 0;
    while (!mbar_try_far(bar, parity)) {
      if ((++spins & 0xFFu) == 0u) {
        if (*abort_flag) { ok = false; break; }
        if ((unsigned long long)(clock64() - t0) > kSpinBudget) { *abort_flag = 1; ok = false; break; }
      }
    }
  }
  return __all_sync(0xffffffffu, ok);
}
// Every lane that looks waits for its own barrier; one verdict for the warp.
__device__ __forceinline__ bool lanes_wait(uint32_t bar, uint32_t parity, bool looks, volatile int *abort_flag) {
  bool there = !looks || mbar_try(bar, parity);
  if (__all_sync(0xffffffffu, there)) return true;
  const unsigned long long t0 = clock64();
  unsigned int spins = 0;
  bool out = false;
  while (!__all_sync(0xffffffffu, there)) {
    if (!there) there = mbar_try(bar, parity);
    if ((++spins & 0xFFu) == 0u) {
      if (*abort_flag) out = true;
      if ((unsigned long long)(clock64() - t0) > kSpinBudget) { *abort_flag = 1; out = true; }
      if (__any_sync(0xffffffffu, out)) return false;
    }
  }
  return true;
}
// For converged warps only: a warp whose lanes arrive in two groups would elect two of them.
__device__ __forceinline__ bool elect_one() {
  uint32_t one;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.b32 %0, 1, 0, p;\n\t}" : "=r"(one));
  return one != 0;
}
__device__ __forceinline__ void mbar_complete_tx(uint32_t bar, uint32_t bytes) {      // as if that many bytes had arrived
  asm volatile("mbarrier.complete_tx.relaxed.cluster.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void st_cluster_u32(uint32_t addr, uint32_t v) {
  asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}
__device__ __forceinline__ uint32_t ld_cluster_u32(uint32_t addr) {
  uint32_t v;
  asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ void st_async_v4(uint32_t addr, uint32_t bar, float a, float b, float c, float d) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%1, %2, %3, %4}, [%5];"
               ::"r"(addr), "f"(a), "f"(b), "f"(c), "f"(d), "r"(bar) : "memory");
}
__device__ __forceinline__ unsigned int ld_acquire(const unsigned int *p) {
  unsigned int v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ bool grid_wait(const unsigned int *word, unsigned int target, volatile int *abort_flag) {
  const unsigned long long t0 = clock64();
  unsigned int spins = 0;
  while (ld_acquire(word) < target)
    if ((++spins & 0x3Fu) == 0u) {
      if (*abort_flag) return false;
      if ((unsigned long long)(clock64() - t0) > kSpinBudget) { *abort_flag = 1; return false; }
    }
  return true;
}
__device__ __forceinline__ void out_meet() { asm volatile("bar.sync 1, 128;" ::: "memory"); }       // the four output warps
// N columns of the high and of the low products.  One statement: the registers hold nothing before the wait, so nothing that
// reads them may be moved between the loads and it.
template <int N>
__device__ __forceinline__ void tmem_ld_pair(uint32_t at_hi, uint32_t at_lo, uint32_t (&hi)[N], uint32_t (&lo)[N]) {
  if constexpr (N == 8) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%16];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%8,%9,%10,%11,%12,%13,%14,%15}, [%17];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=&r"(hi[0]), "=&r"(hi[1]), "=&r"(hi[2]), "=&r"(hi[3]), "=&r"(hi[4]), "=&r"(hi[5]), "=&r"(hi[6]), "=&r"(hi[7]),
          "=&r"(lo[0]), "=&r"(lo[1]), "=&r"(lo[2]), "=&r"(lo[3]), "=&r"(lo[4]), "=&r"(lo[5]), "=&r"(lo[6]), "=&r"(lo[7])
        : "r"(at_hi), "r"(at_lo) : "memory");
  } else {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%32];\n\t"
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%33];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=&r"(hi[0]), "=&r"(hi[1]), "=&r"(hi[2]), "=&r"(hi[3]), "=&r"(hi[4]), "=&r"(hi[5]), "=&r"(hi[6]), "=&r"(hi[7]), "=&r"(hi[8]), "=&r"(hi[9]), "=&r"(hi[10]), "=&r"(hi[11]), "=&r"(hi[12]), "=&r"(hi[13]), "=&r"(hi[14]), "=&r"(hi[15]),
          "=&r"(lo[0]), "=&r"(lo[1]), "=&r"(lo[2]), "=&r"(lo[3]), "=&r"(lo[4]), "=&r"(lo[5]), "=&r"(lo[6]), "=&r"(lo[7]), "=&r"(lo[8]), "=&r"(lo[9]), "=&r"(lo[10]), "=&r"(lo[11]), "=&r"(lo[12]), "=&r"(lo[13]), "=&r"(lo[14]), "=&r"(lo[15])
        : "r"(at_hi), "r"(at_lo) : "memory");
  }
}
__device__ __forceinline__ uint32_t pack_pair(float a, float b) {
  __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<uint32_t *>(&v);
}
__device__ __forceinline__ float lo_of(uint32_t p) { return __uint_as_float(p << 16); }
__device__ __forceinline__ float hi_of(uint32_t p) { return __uint_as_float(p & 0xFFFF0000u); }
// four adjacent values as high + low
__device__ __forceinline__ void store_pair4(__nv_bfloat16 *dst, long long lo_off, const float (&v)[4]) {
  const uint32_t h0 = pack_pair(v[0], v[1]), h1 = pack_pair(v[2], v[3]);
  *reinterpret_cast<uint2 *>(dst) = make_uint2(h0, h1);
  *reinterpret_cast<uint2 *>(dst + lo_off) = make_uint2(pack_pair(v[0] - lo_of(h0), v[1] - hi_of(h0)), pack_pair(v[2] - lo_of(h1), v[3] - hi_of(h1)));
}
}  // namespace

// ------------------------------------------------------------------------------------ embedding rows -> operand pair
// One block per row: the residual, x * gain as a pair, sum x^2; the first block clears the counters of the forward.
__global__ void __launch_bounds__(256) embed_pair_kernel(const int32_t *tokens, const __nv_bfloat16 *emb, const __nv_bfloat16 *gain, float *x,
                                                         __nv_bfloat16 *pan, float *ss, unsigned int *words, int n_words, int d) {
  // In this order: the kernels behind may read cache lengths and cached keys before they wait, so none of them starts before the
  // step in front is complete.
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  __shared__ float part[8];
  const int r = blockIdx.x;
  const __nv_bfloat16 *src = emb + (long long)tokens[r] * d;
  const bool wide = ((unsigned long long)emb & 7u) == 0;
  float sq = 0.f;
  for (int k = threadIdx.x * 4; k < d; k += 256 * 4) {
    float v[4];
    if (wide) {
      const uint2 w = *reinterpret_cast<const uint2 *>(src + k);
      v[0] = lo_of(w.x); v[1] = hi_of(w.x); v[2] = lo_of(w.y); v[3] = hi_of(w.y);
    } else {
#pragma unroll
      for (int i = 0; i < 4; ++i) v[i] = __bfloat162float(src[k + i]);
    }
    *reinterpret_cast<float4 *>(x + (long long)r * d + k) = make_float4(v[0], v[1], v[2], v[3]);
    const uint2 g = __ldg(reinterpret_cast<const uint2 *>(gain + k));
#pragma unroll
    for (int i = 0; i < 4; ++i) sq = fmaf(v[i], v[i], sq);
    v[0] *= lo_of(g.x); v[1] *= hi_of(g.x); v[2] *= lo_of(g.y); v[3] *= hi_of(g.y);
    store_pair4(pan + (long long)r * d + k, (long long)kClusterRows * d, v);
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
  if (r == 0)
    for (int i = threadIdx.x; i < n_words; i += 256) words[i] = 0u;
}

// ------------------------------------------------------------------------------------ projections
template <int BN>
__global__ void __launch_bounds__(kThreadsCl, 1) cluster_chain_kernel(const __grid_constant__ ClMaps maps, const __grid_constant__ ClParams p) {
  using C = ClCfg<BN>;
  constexpr int T = C::T, H = C::H, NACC = C::NACC, NX = C::NX, NCB = C::NCB, S = C::S;
  extern __shared__ unsigned char smem_dyn[];
  __shared__ __align__(8) unsigned long long full_w[S], empty_w[S], full_x[NX], empty_x[NX], acc_full[NACC], acc_empty[NACC], xc_full[C::NXB], xc_empty[C::NXB], drain_bar;
  __shared__ __align__(16) float red[512];         // partial sums of squares; running maxima
  __shared__ float s_row[BN];                      // 1/rms per row
  __shared__ int2 tiles_s[T];                      // warp 0
  __shared__ uint32_t tmem_base_s;
  __shared__ int abort_s, issued_w_s, issued_x_s;
  // Exchange units sent, taken and expected, for the end of a launch in which a wait ran out.  (Branches for it in the exchange's loops, and its
  // code in front of the way out, cost 1 to 4 % of a step: 8 layers of 1.1B, 64 rows 620 us, now 606.)
  __shared__ int sent_s[8], taken_s, expected_s, peer_abort_s;
  const uint32_t base = (smem_u32(smem_dyn) + 1023u) & ~1023u;
  const uint32_t xs_base = base + S * kStageW, xc_base = xs_base + NX * C::kXSlot;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = (int)cluster_rank(), cl = blockIdx.x / kCl;
  volatile int *abort_flag = &abort_s;

  // Tiles of a pass for the thread that requests weights: (first weight row, height in units | index into ClMaps::w << 8).
  auto list_tiles = [&](const Phase &ph, int t0, int t1) {
    int mat, u, h;
    ph.tile(p, min(t0 + lane, t1 - 1), mat, u, h);
    const Kind &k = p.kind[ph.kind];
    const int h0 = ph.kind == PH_QKV && mat > 0 ? p.kv.h0 : k.h0;
    if (lane < T) tiles_s[lane] = make_int2(u * kUnit, h | (2 * (k.mat0 + mat) + h - h0) << 8);
    __syncwarp();
  };
  auto request = [&](const Phase &ph, int st, int t, int pr) {
    const int2 ti = tiles_s[t];
    const int h = ti.y & 0xff;
    const uint32_t bar = smem_u32(&full_w[st]);
    mbar_expect_tx(bar, (uint32_t)h * (2 * kUnit * 128));
    if (h > 0) load_3d(base + st * kStageW, &maps.w[0][0] + (ti.y >> 8), 0, ti.x, 2 * ph.pair(pr), bar);
  };
  // The ring's first round of weights is requested before everything else: the rest of the set-up takes about 3 us (tensor memory,
  // barriers, the cluster's meeting).
  int primed = 0;
  if (warp == 0) {
    const Phase ph = phase_of(p, p.first, cl, rank);
    const int t1 = ph.pass_end<T>(0);
    list_tiles(ph, 0, t1);
    if (lane == 0) {
      for (int i = 0; i < S; ++i) { mbar_init(smem_u32(&full_w[i]), 1); mbar_init(smem_u32(&empty_w[i]), 1); }
      fence_barrier_init();
      fence_proxy_async();                         // the copies below count on them
      for (int t = 0; t < t1; ++t)                 // the first segment of the first pass
        for (int pr = 0; pr < min(2, ph.np) && primed < S; ++pr, ++primed) request(ph, primed, t, pr);
    }
    __syncwarp();
  } else if (warp == 2) {
    // the other barriers, one per lane
    if (lane == 0) { abort_s = 0; peer_abort_s = 0; issued_w_s = 0; issued_x_s = 0; mbar_init(smem_u32(&drain_bar), 1); }
    if (lane < NX) { mbar_init(smem_u32(&full_x[lane]), 1); mbar_init(smem_u32(&empty_x[lane]), 1); }
    if (lane < NACC) { mbar_init(smem_u32(&acc_full[lane]), 1); mbar_init(smem_u32(&acc_empty[lane]), 8); }
    // an exchange buffer is free again when the four output warps of all four CTAs have read theirs
    if (lane < C::NXB) { mbar_init(smem_u32(&xc_full[lane]), 1); mbar_init(smem_u32(&xc_empty[lane]), 4 * kCl); }
    fence_barrier_init();
    if (lane < 3) asm volatile("prefetch.tensormap [%0];" ::"l"(&maps.x[lane]) : "memory");
    __syncwarp();
  }
  if (warp == 1) tmem_alloc(smem_u32(&tmem_base_s), C::kCols);
  tc_fence_before();
  __syncthreads();
  __syncwarp();                                    // the cluster's barrier counts warps
  // The peers' barriers have to exist before anything arrives on them: only the warps that send across the cluster wait for that
  // now (1.5 us that the first activations need not wait), the others before the meeting at the end.
  asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");      // the barriers themselves were released by their fence
  const bool sends = warp >= kDrainWarp0;
  if (sends) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  tc_fence_after();
  const uint32_t tmem_base = tmem_base_s;
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

  if (warp == 0) {
    // ------------------------------------------------------------ weights: wait for nothing but free stages
    int st = 0, issued = 0, ok = 1;
    uint32_t par = 1;
    for (int id = p.first; id < p.last && ok; ++id) {
      const Phase ph = phase_of(p, id, cl, rank);
      for (int t0 = 0, t1; t0 < ph.n_tiles && ok; t0 = t1) {
        t1 = ph.pass_end<T>(t0);
        list_tiles(ph, t0, t1);
        if (lane == 0)
          for (int s = 0; s < ph.np && ok; s += 2)
            for (int t = t0; t < t1 && ok; ++t)
              for (int pr = s; pr < min(s + 2, ph.np); ++pr) {
                if (issued >= primed) {            // the others were requested before the set-up, and may have been used already
                  if (!mbar_wait(smem_u32(&empty_w[st]), par, abort_flag)) { ok = 0; break; }
                  request(ph, st, t - t0, pr);
                }
                ++issued;
                if (++st == S) { st = 0; par ^= 1u; }
              }
        ok = __shfl_sync(0xffffffffu, ok, 0);
      }
    }
    // the MMAs' completions of the last round have landed on this CTA's barriers before it leaves
    if (lane == 0 && ok)
      for (int i = max(0, issued - S); i < issued; ++i)
        if (!mbar_wait(smem_u32(&empty_w[i % S]), (uint32_t)(i / S) & 1u, abort_flag)) break;
    if (lane == 0) issued_w_s = issued;
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer
    // A satisfied wait costs this warp about 200 cycles, sixteen MMAs of N = 32 640: the lanes look at all barriers of a segment
    // at the same time.  (One thread that waits for each on its own: 0.67 us per 32 KB stage, 5 TB/s in all.)
    constexpr uint32_t kIdesc = make_idesc(C::kAcc);
    int st = 0, xpos = 0, use = 0;
    uint32_t par = 0;
    bool ok = true;
    for (int id = p.first; id < p.last && ok; ++id) {
      const Phase ph = phase_of(p, id, cl, rank);
      for (int t0 = 0, t1; t0 < ph.n_tiles && ok; t0 = t1) {
        t1 = ph.pass_end<T>(t0);
        int h_of;                                  // lane i: height of the pass's tile i
        {
          int mat, u;
          ph.tile(p, min(t0 + lane, t1 - 1), mat, u, h_of);
        }
        for (int s = 0; s < ph.np && ok; s += 2) {
          const int n = min(2, ph.np - s);
          for (int t = t0; t < t1 && ok; ++t, ++use) {
            const int h = __shfl_sync(0xffffffffu, h_of, t - t0);
            const int ab = use % NACC;
            const int st1 = st + 1 == S ? 0 : st + 1;
            const uint32_t par1 = st + 1 == S ? par ^ 1u : par;
            const int nx = n * 2 / C::XK;          // activation slots of the segment
            uint32_t bar = smem_u32(&acc_empty[ab]), want = ((uint32_t)(use / NACC) & 1u) ^ 1u;
            if (lane == 1) { bar = smem_u32(&full_w[st]); want = par; }
            if (lane == 2) { bar = smem_u32(&full_w[st1]); want = par1; }
            if (lane >= 3) { const int xi = xpos + lane - 3; bar = smem_u32(&full_x[xi % NX]); want = (uint32_t)(xi / NX) & 1u; }
            const bool looks = lane < 2 || (lane == 2 && n > 1) || (t == t0 && lane >= 3 && lane < 3 + nx);
            ok = lanes_wait(bar, want, looks, abort_flag);
            if (!ok) break;
            tc_fence_after();
            if (elect_one()) {
              const uint32_t d_tmem = tmem_base + (uint32_t)(ab * C::kAcc);
#pragma unroll
              for (int pr = 0; pr < 2; ++pr) {
                if (pr >= n) break;
                const uint32_t wa = base + (pr ? st1 : st) * kStageW;
#pragma unroll
                for (int kb = 0; kb < 2; ++kb) {
                  const int xi = (xpos + (pr * 2 + kb) / C::XK) % NX;
                  const uint64_t ad = smem_desc_sw128(wa + (uint32_t)(kb * h) * (kUnit * 128));
                  const uint64_t bd = smem_desc_sw128(xs_base + (uint32_t)xi * C::kXSlot + (uint32_t)(kb % C::XK) * C::kXBlock);
#pragma unroll
                  for (int kk = 0; kk < kTileK / 16; ++kk)
                    umma_bf16(d_tmem, ad + (uint64_t)(kk * 2), bd + (uint64_t)(kk * 2), kIdesc, (pr > 0 || kb > 0 || kk > 0) ? 1u : 0u);
                  if (t + 1 == t1 && kb % C::XK == C::XK - 1) umma_commit(smem_u32(&empty_x[xi]));
                }
                umma_commit(smem_u32(&empty_w[pr ? st1 : st]));
              }
              umma_commit(smem_u32(&acc_full[ab]));
            }
            __syncwarp();
            for (int i = 0; i < n; ++i)
              if (++st == S) { st = 0; par ^= 1u; }
          }
          xpos += n * 2 / C::XK;
        }
      }
    }
  } else if (warp == 2) {
    // ------------------------------------------------------------ activations
    if (lane == 0) {
      int issued = 0;
      bool ok = true;
      for (int id = p.first; id < p.last && ok; ++id) {
        const Phase ph = phase_of(p, id, cl, rank);
        const CUtensorMap *map = &maps.x[ph.kind == PH_O ? 1 : ph.kind == PH_DOWN ? 2 : 0];
        const unsigned int *word = p.bar + 2 * (id - 1);          // results of the projection in front: [all, first column ranges]
        int seen = 0;                                             // of its two words
        for (int t0 = 0; t0 < ph.n_tiles && ok; t0 = ph.pass_end<T>(t0))
          for (int i = 0; i < ph.np * 2 / C::XK; ++i) {
            const int pr = i * C::XK / 2, sl = issued % NX;
            if (!mbar_wait(smem_u32(&empty_x[sl]), ((uint32_t)(issued / NX) & 1u) ^ 1u, abort_flag)) { ok = false; break; }
            const uint32_t bar = smem_u32(&full_x[sl]);
            mbar_expect_tx(bar, C::kXSlot);
            const int need = ph.kind == PH_DOWN && pr < ph.np0 ? 1 : 2;
            if (seen < need) {
              if (id == p.first) asm volatile("griddepcontrol.wait;" ::: "memory");     // they are the kernel's in front
              else if (!grid_wait(word + (need == 1 ? 1 : 0), p.arrivals, abort_flag)) { ok = false; break; }
              asm volatile("fence.proxy.async.global;" ::: "memory");      // rows stored by other CTAs, read by the TMA
              seen = need;
            }
            load_4d(xs_base + sl * C::kXSlot, map, 0, 0, 0, 2 * ph.pair(pr) + (i * C::XK & 1), bar);
            ++issued;
          }
      }
      for (int i = max(0, issued - NX); i < issued && ok; ++i) ok = mbar_wait(smem_u32(&empty_x[i % NX]), (uint32_t)(i / NX) & 1u, abort_flag);
      issued_x_s = issued;
    }
  } else if (warp < kOutWarp0) {
    // ------------------------------------------------------------ accumulators -> fp32 sums -> the cluster's owners
    const int q = warp & 3, half = (warp - kDrainWarp0) >> 2;     // tensor-memory lanes 32 q .. 32 q + 31, rows half * H ..
    const uint32_t t_lane = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(half * H);
    // weight rows 32 q .. of a tile go to CTA q of the cluster
    const uint32_t dst = map_to_cta(xc_base, (uint32_t)q) + (uint32_t)((rank * 32 + lane) * kXRow * 4);
    const uint32_t dbar = map_to_cta(smem_u32(&xc_full[0]), (uint32_t)q);
    int use = 0, e = 0, sent = 0;                                 // sent: units of this half
    bool ok = true;
    for (int id = p.first; id < p.last && ok; ++id) {
      const Phase ph = phase_of(p, id, cl, rank);
      const int nseg = ph.np > 0 ? (ph.np + 1) >> 1 : 1;          // no share of a short k range: a sum of zero is sent
      for (int t0 = 0, tn; t0 < ph.n_tiles && ok; t0 += tn) {
        tn = ph.pass_end<T>(t0) - t0;
        float sum[T][H];
#pragma unroll
        for (int t = 0; t < T; ++t)
#pragma unroll
          for (int i = 0; i < H; ++i) sum[t][i] = 0.f;
        for (int sg = 0; sg < nseg && ok; ++sg) {
#pragma unroll
          for (int t = 0; t < T; ++t) {
            if (t >= tn || !ok) continue;
            if (ph.np > 0) {
              const int ab = use % NACC;
              ok = mbar_wait_warp(smem_u32(&acc_full[ab]), (uint32_t)(use / NACC) & 1u, abort_flag);
              if (!ok) continue;
              tc_fence_after();
              const uint32_t ta = t_lane + (uint32_t)(ab * C::kAcc);
              constexpr int N = H < 16 ? 8 : 16;
#pragma unroll
              for (int j = 0; j < H; j += N) {
                uint32_t hi[N], lo[N];
                tmem_ld_pair<N>(ta + j, ta + BN + j, hi, lo);
#pragma unroll
                for (int i = 0; i < N; ++i) sum[t][j + i] += __uint_as_float(hi[i]) + __uint_as_float(lo[i]);
              }
              tc_fence_before();
              __syncwarp();
              if (lane == 0) mbar_arrive(smem_u32(&acc_empty[ab]));
              ++use;
            }
            if (sg + 1 == nseg) {
#pragma unroll
              for (int cb = 0; cb < NCB; ++cb) {
                if (BN > 16 && cb / (NCB / 2 > 0 ? NCB / 2 : 1) != half) continue;       // the other half's rows
                const int u = e + t * NCB + cb, b = u % C::NXB;
                if (u >= C::NXB && ok) {
                  ok = wait_far(smem_u32(&xc_empty[b]), (uint32_t)(u / C::NXB - 1) & 1u, abort_flag);
                }
                if (!ok) continue;
                const uint32_t to = dst + (uint32_t)(b * kXBuf), bar = dbar + (uint32_t)b * 8u;
                constexpr int N = H < 16 ? H : 16;
                const float *v = &sum[t][BN > 16 ? (cb % (NCB / 2 > 0 ? NCB / 2 : 1)) * 16 : 0];
                sent += 1;
#pragma unroll
                for (int i = 0; i < N; i += 4) st_async_v4(to + (uint32_t)((BN > 16 ? 0 : half * H) + i) * 4u, bar, v[i], v[i + 1], v[i + 2], v[i + 3]);
              }
            }
          }
        }
        e += tn * NCB;
      }
    }
    if (lane == 0) sent_s[warp - kDrainWarp0] = sent;
    // the peers' arrivals of the last units too: one that lands in the next kernel's barrier would let a sender there go too early
    for (int u = max(0, e - C::NXB); u < e && ok; ++u)
      if (BN == 16 || (u % NCB) / (NCB / 2 > 0 ? NCB / 2 : 1) == half) ok = wait_far(smem_u32(&xc_empty[u % C::NXB]), (uint32_t)(u / C::NXB) & 1u, abort_flag);
  } else {
    // ------------------------------------------------------------ finished values
    const int ot = threadIdx.x - kOutWarp0 * 32, n = ot & 15, mq = ot >> 4;       // row n of a block of 16, weight rows 4 mq .. 4 mq + 3 of this CTA's 32
    const unsigned char *xc_gen = smem_dyn + (xc_base - smem_u32(smem_dyn));
    const uint32_t far_empty = map_to_cta(smem_u32(&xc_empty[0]), (uint32_t)(lane & 3));
    const bool wide_logits = ((unsigned long long)p.logits & 15u) == 0;
    int e = 0;
    bool ok = true;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    for (int id = p.first; id < p.last; ++id) {
      const Phase ph = phase_of(p, id, cl, rank);
      const int kind = ph.kind;
      if (id != p.first && ot == 0) (void)grid_wait(p.bar + 2 * (id - 1), p.arrivals, abort_flag);
      out_meet();
      if (kind == PH_GU || kind == PH_HEAD || (kind == PH_QKV && blockIdx.x == 0)) {
        // row sums of squares over the slots of all CTAs, in a fixed order
        const float *ss = kind == PH_GU ? p.ss_ffn : p.ss_x;
        const int slots = id == 0 ? p.first_slots : (int)gridDim.x;
        constexpr int W = BN / 4, G = 128 / W;
        float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int i = ot / W; i < slots; i += G) {
          const float4 v = __ldcg(reinterpret_cast<const float4 *>(ss + (size_t)i * kClusterRows) + ot % W);
          a.x += v.x; a.y += v.y; a.z += v.z; a.w += v.w;
        }
        reinterpret_cast<float4 *>(red)[ot] = a;
        out_meet();
        if (ot < BN) {
          float t = 0.f;
          for (int i = 0; i < G; ++i) t += red[i * BN + ot];
          if (kind == PH_QKV) { if (ot < p.R) p.ss_attn[ot] = t; }
          else s_row[ot] = rsqrtf(t / (float)p.dn + p.eps);
        }
        out_meet();
      }
      float sq[NCB], gate[NCB][4];
      unsigned long long best[NCB];
      int bias_at[NCB];
#pragma unroll
      for (int cb = 0; cb < NCB; ++cb) {
        sq[cb] = 0.f; best[cb] = 0ull; bias_at[cb] = -1;
        if (kind == PH_HEAD && p.perm && cb * 16 + n < p.R) bias_at[cb] = p.perm[p.tokens[cb * 16 + n]];
#pragma unroll
        for (int i = 0; i < 4; ++i) gate[cb][i] = 0.f;
      }
      auto publish = [&](unsigned int *word) {
        asm volatile("fence.proxy.async.global;" ::: "memory");   // generic stores in front of other CTAs' TMA reads
        out_meet();
        if (ot == 0) asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(word), "r"(1u) : "memory");
      };
      for (int t = 0; t < ph.n_tiles; ++t) {
        if (t == ph.early && t > 0) publish(p.bar + 2 * id + 1);
        int mat, u, h;
        ph.tile(p, t, mat, u, h);
        const int m0 = rank * 32 + mq * 4, col = u * kUnit + m0;
        const bool live = m0 < h * kUnit;
        const __nv_bfloat16 *gain = kind == PH_O ? p.g_ffn : p.g_next;
        uint2 gq = make_uint2(0u, 0u);
        if (live && (kind == PH_O || kind == PH_DOWN)) gq = __ldg(reinterpret_cast<const uint2 *>(gain + col));
#pragma unroll
        for (int cb = 0; cb < NCB; ++cb, e += ok) {      // a wait that ran out: e stays at its unit
          const int r = cb * 16 + n, b = e % C::NXB;
          const bool mine = live && r < p.R;
          float4 xr = make_float4(0.f, 0.f, 0.f, 0.f);
          if (mine && (kind == PH_O || kind == PH_DOWN)) xr = __ldcg(reinterpret_cast<const float4 *>(p.x + (long long)r * p.d + col));
          if (ok && ot == 0) mbar_expect_tx(smem_u32(&xc_full[b]), kXBuf);
          if (ok) {
            ok = wait_far(smem_u32(&xc_full[b]), (uint32_t)(e / C::NXB) & 1u, abort_flag);
          }
          if (!ok) continue;
          const float *src = reinterpret_cast<const float *>(xc_gen + b * kXBuf) + (mq * 4) * kXRow + n;
          float v[4];
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            v[i] = src[i * kXRow];
#pragma unroll
            for (int k = 1; k < kCl; ++k) v[i] += src[(k * 32 + i) * kXRow];
          }
          // the buffer is free: every lane's loads are in front of the arrival (a barrier of the warp, then the release)
          __syncwarp();
          if (lane < kCl) mbar_arrive_far(far_empty + (uint32_t)b * 8u);
          if (kind == PH_O || kind == PH_DOWN) {
            if (mine) {
              v[0] += xr.x; v[1] += xr.y; v[2] += xr.z; v[3] += xr.w;
              *reinterpret_cast<float4 *>(p.x + (long long)r * p.d + col) = make_float4(v[0], v[1], v[2], v[3]);
#pragma unroll
              for (int i = 0; i < 4; ++i) sq[cb] = fmaf(v[i], v[i], sq[cb]);
              v[0] *= lo_of(gq.x); v[1] *= hi_of(gq.x); v[2] *= lo_of(gq.y); v[3] *= hi_of(gq.y);
              store_pair4(p.pan_x + (long long)r * p.d + col, (long long)kClusterRows * p.d, v);
            }
          } else if (kind == PH_GU) {
            if (mat == 0) {
#pragma unroll
              for (int i = 0; i < 4; ++i) gate[cb][i] = v[i];
            } else if (mine) {
              const float s = s_row[r];
#pragma unroll
              for (int i = 0; i < 4; ++i) {
                const float g = s * gate[cb][i];
                v[i] = __fdividef(g, 1.0f + __expf(-g)) * (s * v[i]);
              }
              store_pair4(p.pan_h + (long long)r * p.f + col, (long long)kClusterRows * p.f, v);
            }
          } else if (kind == PH_QKV) {
            if (mine) {
              const int at = (mat == 0 ? 0 : mat == 1 ? p.qd : p.qd + p.kvd) + col;
              *reinterpret_cast<float4 *>(p.qkv + (long long)r * (p.qd + 2 * p.kvd) + at) = make_float4(v[0], v[1], v[2], v[3]);
            }
          } else if (mine) {
            const float s = s_row[r];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              v[i] *= s;
              if (bias_at[cb] == col + i) v[i] += p.beta;
              const unsigned long long key = ((unsigned long long)ordered_key_u(v[i]) << 32) | (unsigned long long)(0xFFFFFFFFu - (unsigned int)(col + i));
              best[cb] = key > best[cb] ? key : best[cb];
            }
            if (p.logits) {
              float *lp = p.logits + (long long)r * p.vocab + col;
              if (wide_logits) *reinterpret_cast<float4 *>(lp) = make_float4(v[0], v[1], v[2], v[3]);
              else { lp[0] = v[0]; lp[1] = v[1]; lp[2] = v[2]; lp[3] = v[3]; }
            }
          }
        }
      }
      if (kind == PH_O || kind == PH_DOWN) {
        // this CTA's slot of the row sums of squares
#pragma unroll
        for (int cb = 0; cb < NCB; ++cb) {
          const float v = sq[cb] + __shfl_xor_sync(0xffffffffu, sq[cb], 16);
          if (lane < 16) red[(ot >> 5) * BN + cb * 16 + lane] = v;
        }
        out_meet();
        if (ot < BN) (kind == PH_O ? p.ss_ffn : p.ss_x)[(size_t)blockIdx.x * kClusterRows + ot] = red[ot] + red[BN + ot] + red[2 * BN + ot] + red[3 * BN + ot];
      } else if (kind == PH_HEAD) {
        unsigned long long *rk = reinterpret_cast<unsigned long long *>(red);
#pragma unroll
        for (int cb = 0; cb < NCB; ++cb) {
          const unsigned long long o = __shfl_xor_sync(0xffffffffu, best[cb], 16), v = best[cb] > o ? best[cb] : o;
          if (lane < 16) rk[(ot >> 5) * BN + cb * 16 + lane] = v;
        }
        out_meet();
        if (ot < BN && ot < p.R) {
          unsigned long long v = rk[ot];
#pragma unroll
          for (int w = 1; w < 4; ++w) v = rk[w * BN + ot] > v ? rk[w * BN + ot] : v;
          if (v) atomicMax(&p.amax[ot], v);
        }
      }
      if (id + 1 < p.last) publish(p.bar + 2 * id);
    }
    if (ot == 0) { taken_s = e; expected_s = e + !ok; }
    asm volatile("fence.proxy.async.global;" ::: "memory");       // for the TMA reads of the next kernel
  }

  // ---------------------------------------------------------------- teardown
  __syncwarp();
  if (!sends) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  __syncthreads();
  if (abort_s) {
    if (threadIdx.x == 0) {
      atomicExch(p.err, 1u);
      for (int r = 0; r < kCl; ++r) st_cluster_u32(map_to_cta(smem_u32(&peer_abort_s), (uint32_t)r), 1u);
      const unsigned long long t0 = clock64();                    // copies still in flight (bounded)
      for (int i = max(0, issued_w_s - S); i < issued_w_s; ++i)
        while (!mbar_try(smem_u32(&full_w[i % S]), (uint32_t)(i / S) & 1u))
          if ((unsigned long long)(clock64() - t0) > kSpinBudget / 4) break;
      for (int i = max(0, issued_x_s - NX); i < issued_x_s; ++i)
        while (!mbar_try(smem_u32(&full_x[i % NX]), (uint32_t)(i / NX) & 1u))
          if ((unsigned long long)(clock64() - t0) > kSpinBudget / 4) break;
    }
    __syncwarp();
    if (warp == 1 && elect_one()) {
      umma_commit(smem_u32(&drain_bar));
      const unsigned long long t0 = clock64();
      while (!mbar_try(smem_u32(&drain_bar), 0u))
        if ((unsigned long long)(clock64() - t0) > kSpinBudget / 4) break;
    }
    __syncthreads();
    asm volatile("fence.acq_rel.cluster;" ::: "memory");      // the peers' flags, in front of the closing barrier
  }
  tc_fence_before();
  __syncthreads();
  __syncwarp();
  // No CTA leaves while a peer may still write to it.  (Relaxed: what goes across the cluster has been waited for above; a release would
  // also wait for the last global stores, which the end of the grid does.)
  asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, C::kCols);
  }
  if (__builtin_expect(*(volatile int *)&peer_abort_s, 0)) {
    // A wait ran out in this cluster, so not everything that was sent has been waited for.  Every CTA learns from its peers how far
    // they sent, lets each buffer expect that and no more, and waits (bounded) for it to land.
    cluster_sync_all();
    if (threadIdx.x == 0) {
      const unsigned long long t0 = clock64();
#pragma unroll 1
      for (int b = 0; b < C::NXB; ++b) {
        int u = taken_s;                                          // the first unit of this buffer that was not taken
        while (u % C::NXB != b) ++u;
        const int u_half = BN == 16 ? u : u / NCB * (NCB / 2) + u % (NCB / 2 > 0 ? NCB / 2 : 1);      // its number among a half's units
        uint32_t bytes = 0;
#pragma unroll 1
        for (int r = 0; r < kCl; ++r)
#pragma unroll 1
          for (int w = 0; w < 8; ++w)                             // the senders whose weight rows are this CTA's
            if (((w + kDrainWarp0) & 3) == rank && u_half < (int)ld_cluster_u32(map_to_cta(smem_u32(&sent_s[w]), (uint32_t)r)) &&
                (BN == 16 || (u % NCB) / (NCB / 2 > 0 ? NCB / 2 : 1) == w >> 2))
              bytes += 32 * (BN == 16 ? H : 16) * 4;
        const uint32_t bar = smem_u32(&xc_full[b]);
        if (u < expected_s) { if (bytes < (uint32_t)kXBuf) mbar_complete_tx(bar, (uint32_t)kXBuf - bytes); }
        else if (bytes > 0) mbar_expect_tx(bar, bytes);
        else continue;
        while (!mbar_try(bar, (uint32_t)(u / C::NXB) & 1u))
          if ((unsigned long long)(clock64() - t0) > kSpinBudget / 4) break;
      }
    }
    __syncthreads();
    __syncwarp();
    cluster_sync_all();
  }
}

// ------------------------------------------------------------------------------------ host side
typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
static EncodeTiledFn encode_fn() {
  static EncodeTiledFn enc = nullptr;
  if (!enc) {
    void *sym = nullptr;
    cudaDriverEntryPointQueryResult qres;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &sym, cudaEnableDefault, &qres) != cudaSuccess || qres != cudaDriverEntryPointSuccess) return nullptr;
    enc = (EncodeTiledFn)sym;
  }
  return enc;
}

struct ClusterPlan {
  ClusterModel m;
  int ncl;
  double fill;                                     // stage_fill() of a layer
  long long layer_bytes;
  Kind kind[5], kv;
  ClMaps maps[3];                                  // operand boxes of 16, 32, 64 rows; the weights' are filled in per launch
  std::vector<std::array<CUtensorMap, 2>> w;       // [layer][kMats], then the LM head
};

template <int BN>
static cudaError_t cluster_config(cudaLaunchConfig_t &cfg, cudaLaunchAttribute (&attr)[2], int ncl, int pdl, cudaStream_t st) {
  static bool attr_done[kMaxDevices] = {false};
  const int dev = current_device_slot();
  if (!attr_done[dev]) {
    cudaError_t e = cudaFuncSetAttribute(cluster_chain_kernel<BN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ClCfg<BN>::kSmem);
    if (e != cudaSuccess) return e;
    attr_done[dev] = true;
  }
  memset(&cfg, 0, sizeof cfg);
  cfg.gridDim = dim3(ncl * kCl); cfg.blockDim = dim3(kThreadsCl); cfg.dynamicSmemBytes = ClCfg<BN>::kSmem; cfg.stream = st;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = kCl; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr; cfg.numAttrs = pdl ? 2 : 1;
  return cudaSuccess;
}
// most = min(most, clusters that run at the same time)
template <int BN>
static cudaError_t cluster_fit(int &most) {
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr[2];
  int n = 0;
  cudaError_t e = cluster_config<BN>(cfg, attr, 1, 0, nullptr);
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveClusters(&n, cluster_chain_kernel<BN>, &cfg);
  if (e == cudaSuccess && n < most) most = n;
  return e;
}

bool cluster_shape_ok(int d, int qd, int kvd, int f, int vocab) {
  for (int n : {d, qd, kvd, f, vocab})
    if (!ranges_exact(n / kUnit, kFewestClusters, kTileUnits)) return false;
  return d % 128 == 0 && qd % 128 == 0 && f % 128 == 0 && kvd % kUnit == 0 && vocab % kUnit == 0;
}

// Pairs: [2][kClusterRows][d | qd | f].  *out is null where the device holds too few of the clusters; anything else that fails is an error.
cudaError_t cluster_plan_create(const ClusterModel &m, void *pan_x, void *pan_a, void *pan_h, ClusterPlan **out) {
  *out = nullptr;
  EncodeTiledFn enc = encode_fn();
  if (!enc || !cluster_shape_ok(m.d, m.qd, m.kvd, m.f, m.vocab)) return cudaErrorNotSupported;
  int ncl = kClusterSlots / kCl;
  cudaError_t e = cluster_fit<16>(ncl);
  if (e == cudaSuccess) e = cluster_fit<32>(ncl);
  if (e == cudaSuccess) e = cluster_fit<64>(ncl);
  if (e != cudaSuccess || ncl < kFewestClusters) return e;
  ClusterPlan *pl = new (std::nothrow) ClusterPlan();
  if (!pl) return cudaErrorMemoryAllocation;
  pl->m = m; pl->ncl = ncl;
  const int shape[7][2] = {{m.qd, m.d}, {m.kvd, m.d}, {m.kvd, m.d}, {m.d, m.qd}, {m.f, m.d}, {m.f, m.d}, {m.d, m.f}};
  pl->fill = stage_fill(shape, 7, ncl);
  pl->layer_bytes = 2ll * m.d * (2ll * m.qd + 2ll * m.kvd + 3ll * m.f);
  pl->w.resize((size_t)m.n_layers * kMats + 1);
  memset((void *)pl->w.data(), 0, pl->w.size() * sizeof pl->w[0]);
  bool ok = true;
  auto kind_of = [&](int N, int K, int mat0) {
    Kind k; memset(&k, 0, sizeof k);
    k.units = N / kUnit; k.parts = k.n_tiles = column_ranges(k.units, ncl, kTileUnits); k.inv_parts = reciprocal(k.parts);
    k.pairs = k.first = K >> 7; k.mat0 = mat0;
    k.h0 = k.units / k.parts / ncl;                // ranges differ by one unit, and so do the tiles of a range
    return k;
  };
  pl->kv = kind_of(m.kvd, m.d, 0);
  pl->kind[PH_QKV] = kind_of(m.qd, m.d, 0); pl->kind[PH_QKV].n_tiles += 2 * pl->kv.parts;
  pl->kind[PH_O] = kind_of(m.d, m.qd, 3);
  Kind &gu = pl->kind[PH_GU] = kind_of(m.f, m.d, 4);
  gu.n_tiles = 2 * gu.parts; gu.early = 2 * (gu.parts - 1);
  pl->kind[PH_DOWN] = kind_of(m.d, m.f, 6);
  pl->kind[PH_DOWN].first = (gu.parts - 1) * gu.units / gu.parts * kUnit >> 7;
  pl->kind[PH_HEAD] = kind_of(m.vocab, m.d, 0);
  auto weight_maps = [&](std::array<CUtensorMap, 2> &out, const void *w, int N, int K) {
    const int h0 = kind_of(N, K, 0).h0;
    for (int h = h0 > 1 ? h0 : 1; h <= h0 + 1 && h <= kTileUnits && ok; ++h) {
      cuuint64_t gdim[3] = {64, (cuuint64_t)N, (cuuint64_t)K / 64}, gstr[2] = {(cuuint64_t)K * 2, 128};
      cuuint32_t box[3] = {64, (cuuint32_t)(h * kUnit), 2}, estr[3] = {1, 1, 1};
      ok = enc(&out[h - h0], CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void *>(w), gdim, gstr, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
               CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
    }
  };
  for (int l = 0; l < m.n_layers && ok; ++l) {
    std::array<CUtensorMap, 2> *o = pl->w.data() + (size_t)l * kMats;
    weight_maps(o[0], m.wq[l], m.qd, m.d);
    weight_maps(o[1], m.wk[l], m.kvd, m.d);
    weight_maps(o[2], m.wv[l], m.kvd, m.d);
    weight_maps(o[3], m.wo[l], m.d, m.qd);
    weight_maps(o[4], m.w_gate[l], m.f, m.d);
    weight_maps(o[5], m.w_up[l], m.f, m.d);
    weight_maps(o[6], m.w_down[l], m.d, m.f);
  }
  weight_maps(pl->w.back(), m.lm_head, m.vocab, m.d);
  void *pans[3] = {pan_x, pan_a, pan_h};
  const int ks[3] = {m.d, m.qd, m.f};
  for (int b = 0; b < 3; ++b)
    for (int i = 0; i < 3 && ok; ++i) {
      const cuuint64_t K = (cuuint64_t)ks[i];
      cuuint64_t gdim[4] = {64, (cuuint64_t)kClusterRows, 2, K / 64}, gstr[3] = {K * 2, K * 2 * kClusterRows, 128};
      cuuint32_t box[4] = {64, (cuuint32_t)(16 << b), 2, (cuuint32_t)(b == 2 ? ClCfg<64>::XK : ClCfg<16>::XK)}, estr[4] = {1, 1, 1, 1};
      ok = enc(&pl->maps[b].x[i], CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, pans[i], gdim, gstr, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
               CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
    }
  if (!ok) { delete pl; return cudaErrorInvalidValue; }
  *out = pl;
  return cudaSuccess;
}
void cluster_plan_destroy(ClusterPlan *p) { delete p; }
bool cluster_pays(const ClusterPlan *pl, int R, int max_len, bool fused) {
  return pl && R <= kClusterRows && one_writer_pays(pl->fill, pl->layer_bytes, R, max_len, fused);
}

cudaError_t launch_embed_pair(const int32_t *tokens, const void *emb, const void *gain, float *x, void *pan, float *ss, unsigned int *words, int n_words,
                              int R, int d, int pdl, cudaStream_t st) {
  if (R < 1 || R > kClusterRows || d % 4) return cudaErrorInvalidValue;
  cudaLaunchConfig_t cfg;
  memset(&cfg, 0, sizeof cfg);
  cfg.gridDim = dim3(R); cfg.blockDim = dim3(256); cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr; cfg.numAttrs = pdl ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, embed_pair_kernel, tokens, (const __nv_bfloat16 *)emb, (const __nv_bfloat16 *)gain, x, (__nv_bfloat16 *)pan, ss, words, n_words, d);
}

template <int BN>
static cudaError_t launch_cluster_t(const ClMaps &maps, const ClParams &p, int ncl, int pdl, cudaStream_t st) {
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr[2];
  cudaError_t e = cluster_config<BN>(cfg, attr, ncl, pdl, st);
  return e == cudaSuccess ? cudaLaunchKernelEx(&cfg, cluster_chain_kernel<BN>, maps, p) : e;
}

cudaError_t launch_cluster_chain(const ClusterPlan *pl, const ClusterArgs &a, int first, int last, int pdl, cudaStream_t st) {
  const ClusterModel &m = pl->m;
  if (a.R < 1 || a.R > kClusterRows || first < 0 || first >= last || last > 4 * m.n_layers + 1 || last - first > 4) return cudaErrorInvalidValue;
  ClParams p;
  memset(&p, 0, sizeof p);
  memcpy(p.kind, pl->kind, sizeof p.kind);
  p.kv = pl->kv; p.inv_ncl = reciprocal(pl->ncl);
  p.first = first; p.last = last; p.n_layers = m.n_layers; p.d = m.d; p.qd = m.qd; p.kvd = m.kvd; p.f = m.f; p.vocab = m.vocab; p.R = a.R;
  p.x = a.x; p.qkv = a.qkv; p.pan_x = (__nv_bfloat16 *)a.pan_x; p.pan_h = (__nv_bfloat16 *)a.pan_h;
  p.g_ffn = (const __nv_bfloat16 *)a.g_ffn; p.g_next = (const __nv_bfloat16 *)a.g_next;
  p.ss_x = a.ss_x; p.ss_ffn = a.ss_ffn; p.ss_attn = a.ss_attn; p.first_slots = 1;
  p.eps = a.eps; p.dn = m.d; p.bar = a.bar; p.arrivals = (unsigned int)(pl->ncl * kCl + a.withheld); p.err = a.err;
  p.tokens = a.tokens; p.perm = a.perm; p.beta = a.beta; p.amax = a.amax; p.logits = a.logits;
  const int width = a.R <= 16 ? 0 : a.R <= 32 ? 1 : 2;
  ClMaps maps = pl->maps[width];
  for (int id = first; id < last; ++id) {          // every matrix at most once in four projections
    const int l = id >> 2, kind = l == m.n_layers ? (int)PH_HEAD : id & 3, mat0 = pl->kind[kind].mat0;
    const int n = kind == PH_QKV ? 3 : kind == PH_GU ? 2 : 1;
    for (int i = 0; i < n; ++i) memcpy(maps.w[mat0 + i], &pl->w[(size_t)l * kMats + mat0 + i], sizeof maps.w[0]);
  }
  if (width == 0) return launch_cluster_t<16>(maps, p, pl->ncl, pdl, st);
  if (width == 1) return launch_cluster_t<32>(maps, p, pl->ncl, pdl, st);
  return launch_cluster_t<64>(maps, p, pl->ncl, pdl, st);
}

}  // namespace fc
