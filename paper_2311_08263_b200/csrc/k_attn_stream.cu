// Window attention as a stream over the K/V cache (bf16, head_dim 64/128), for rows whose own K/V are already in it, and
// the kernel in front of it that turns the fp32 QKV accumulators into rotated queries and cache rows.
//
// qkv_finish_kernel: per row the deferred 1/rms factor, the rotation, q as a bf16 pair high + low (in the order of MMA
// operands), k and v as bf16 at their cache slots.
//
// attn_stream_kernel: grid (key splits, kv heads x query groups, segments); a segment is a run of rows of one sequence.
// Three or four consumer warps and one producer thread, two CTAs per SM.  A consumer warp owns 16 query rows and whole tiles of
// 32 keys: scores, probabilities and the 16 x hd output stay in its registers (the accumulators of Q.K^T are the A
// operand of P.V as they are), so a tile needs no CTA barrier and no exchange between warps.  WQ query tiles share
// every key tile of the ring, groups of WQ warps take turns at the tiles: one query tile per kv head (plain decoding,
// small windows) -> three tiles of keys in work at once; 64 rows and more (prompts) -> four query tiles on each key tile.
// The groups' partial results are merged through shared memory, the key splits (one cluster) through distributed
// shared memory.  q and the probabilities enter the tensor cores as bf16 pairs, so that only the stored K/V are rounded.
//
// What bounds it: at one to sixteen query rows per kv head the K/V stream out of HBM; each CTA keeps 96 KB of tiles in
// flight, two CTAs 192 KB per SM.  With many rows it is the mma.sync rate.
// Every wait is bounded: on expiry the error word is set and the CTA goes straight to its barriers.
#include <cstring>

#include "fc_attn.cuh"
#include "fc_internal.h"
#include "fc_plan.h"
#include "fc_ptx.cuh"

namespace fc {

namespace {

constexpr int kSKeys = 32;             // keys per tile
// Consumer warps.  The groups that take turns at the tiles have to divide the ring: a parity wait is only unambiguous for
// a warp that consumes every phase of the stages it waits on.  So one query tile is worked on by three groups, not four.
__host__ __device__ constexpr int stream_warps(int wq) { return wq == 1 ? 3 : 4; }
__host__ __device__ constexpr int stream_threads(int wq) { return (stream_warps(wq) + 1) * 32; }

template <int HD>
struct StreamCfg {
  static constexpr int SUB = HD / 64;                        // 128-byte sub-tiles per row
  static constexpr uint32_t kSub = kSKeys * 128;             // one sub-tile: 32 keys x 128 bytes
  static constexpr uint32_t kHalf = SUB * kSub;              // K (or V) of a tile
  static constexpr uint32_t kTile = 2 * kHalf;
  static constexpr int S = HD == 128 ? 6 : 12;               // 96 KB of tiles
  static constexpr int OLD = HD + 8;                         // row pitch of the partial outputs (floats): spreads the banks
  static constexpr size_t smem() { return 1024 + (size_t)S * kTile; }
};

// Byte offset of 16-byte piece `ch` of key `r` in a tile of 128-byte sub-tiles with the TMA's 128-byte swizzle.
__device__ __forceinline__ uint32_t soff(int r, int ch) {
  return (uint32_t)(ch >> 3) * (kSKeys * 128u) + (uint32_t)r * 128u + (uint32_t)(((ch & 7) ^ (r & 7)) << 4);
}
// Rows of segment i: sequence, first row, number of rows.
__device__ __forceinline__ void seg_of(const RowSegs &g, int i, int &b, int &row0, int &nrows) {
  if (g.n > 0) { b = g.seq[i]; row0 = g.row0[i]; nrows = g.row0[i + 1] - row0; }
  else { b = g.seq_map ? g.seq_map[i] : g.b0 + i; row0 = i * g.c; nrows = g.c; }
}

// Queries are stored tile by tile (16 queries of a kv head, q = row * group + head of the group) in the order in which
// a warp holds them as MMA A operands: [kv head][tile][high, low][16-wide k block][lane][4 registers], so that a warp
// loads a k block with one 16-byte load per lane.  Index in units of 128 registers.
__device__ __forceinline__ long long q_frag(int kvh, int tiles, int tile, int part, int ks, int hd) {
  return (((long long)kvh * tiles + tile) * 2 + part) * (hd >> 4) + ks;
}
// First tile of segment i (each segment starts a tile of its own).
__device__ __forceinline__ int seg_tile0(int row0, int group, int i) { return row0 * group / 16 + i; }

}  // namespace

// ------------------------------------------------------------------------------------ QKV accumulators -> q, K, V
// A thread takes four adjacent pairs (i, i + hd/2) of one head of one row: 16-byte loads, 8-byte stores.  Blocks of a
// row split its heads when there are fewer rows than SMs.
__global__ void __launch_bounds__(256) qkv_finish_kernel(const __grid_constant__ QkvFinishArgs a) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int r = blockIdx.x;
  int b, row0, nrows, sg = 0;
  if (a.segs.n > 0) {
    while (sg + 1 < a.segs.n && r >= a.segs.row0[sg + 1]) ++sg;
  } else {
    sg = r / a.segs.c;
  }
  seg_of(a.segs, sg, b, row0, nrows);
  const int group = a.hq / a.hkv, tile0 = seg_tile0(row0, group, sg);
  const int pos = a.kv_len[b] + (r - row0);
  const int half = a.hd >> 1, per_head = half >> 2;                 // units of four pairs
  const int units = (a.hq + 2 * a.hkv) * per_head;
  const float s = rsqrtf(__ldcg(a.ss + r) / (float)a.dn + a.eps);
  const float *src = a.qkv + (long long)r * a.ldq;
  for (int u = blockIdx.y * 256 + threadIdx.x; u < units; u += gridDim.y * 256) {
    const int h = u / per_head, i = (u - h * per_head) << 2;
    const float *p = src + h * a.hd + i;
    const float4 x = __ldcg(reinterpret_cast<const float4 *>(p)), y = __ldcg(reinterpret_cast<const float4 *>(p + half));
    float v0[4] = {x.x * s, x.y * s, x.z * s, x.w * s}, v1[4] = {y.x * s, y.y * s, y.z * s, y.w * s};
    if (h < a.hq + a.hkv) {
      const float4 *rp = reinterpret_cast<const float4 *>(a.rope + (long long)pos * half + i);
      const float4 c0 = __ldg(rp), c1 = __ldg(rp + 1);
      const float cs[4] = {c0.x, c0.z, c1.x, c1.z}, sn[4] = {c0.y, c0.w, c1.y, c1.w};
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const float o0 = v0[k] * cs[k] - v1[k] * sn[k], o1 = v0[k] * sn[k] + v1[k] * cs[k];
        v0[k] = o0; v1[k] = o1;
      }
    }
    const uint2 h0 = make_uint2(pack2(v0[0], v0[1]), pack2(v0[2], v0[3])), h1 = make_uint2(pack2(v1[0], v1[1]), pack2(v1[2], v1[3]));
    if (h < a.hq) {
      // fragment order (see q_frag): the four elements are one register of two neighbouring lanes
      const int kvh = h / group, q = (r - row0) * group + h - kvh * group, rr = q & 15;
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const int k = i + e * half, kk = k & 15;
        uint32_t *dst = (uint32_t *)a.q + q_frag(kvh, a.q_tiles, tile0 + (q >> 4), 0, k >> 4, a.hd) * 128 + ((rr & 7) * 4 + ((kk & 7) >> 1)) * 4 + (rr >> 3) + 2 * (kk >> 3);
        uint32_t *low = dst + (a.hd >> 4) * 128;
        const uint2 hv = e ? h1 : h0;
        const float *v = e ? v1 : v0;
        dst[0] = hv.x; dst[4] = hv.y;
        low[0] = pack2(v[0] - low_half(hv.x), v[1] - high_half(hv.x));
        low[4] = pack2(v[2] - low_half(hv.y), v[3] - high_half(hv.y));
      }
    } else {
      const bool is_k = h < a.hq + a.hkv;
      const int kvh = h - a.hq - (is_k ? 0 : a.hkv);
      __nv_bfloat16 *dst = (__nv_bfloat16 *)(is_k ? a.kcache : a.vcache) + (long long)b * a.stride_b + (long long)kvh * a.stride_h + (long long)pos * a.hd + i;
      *reinterpret_cast<uint2 *>(dst) = h0;
      *reinterpret_cast<uint2 *>(dst + half) = h1;
    }
  }
  // side clearing: buffers the previous kernel has finished with and a later one accumulates into
  const unsigned long long gtid = ((unsigned long long)blockIdx.y * gridDim.x + blockIdx.x) * 256 + threadIdx.x;
  const unsigned long long nth = (unsigned long long)gridDim.x * gridDim.y * 256;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    if (!a.z.p[i]) continue;
    const unsigned long long n4 = a.z.n[i] >> 2;
    float4 *p4 = reinterpret_cast<float4 *>(a.z.p[i]);
    for (unsigned long long e = gtid; e < n4; e += nth) p4[e] = make_float4(0.f, 0.f, 0.f, 0.f);
    for (unsigned long long e = (n4 << 2) + gtid; e < a.z.n[i]; e += nth) a.z.p[i][e] = 0.f;
  }
}

// ------------------------------------------------------------------------------------ attention
template <int HD, int WQ>
__global__ void __launch_bounds__(stream_threads(WQ), 2)
attn_stream_kernel(const __grid_constant__ CUtensorMap map, const __grid_constant__ StreamAttnArgs a) {
  using C = StreamCfg<HD>;
  constexpr int kSWarps = stream_warps(WQ), kSThreads = stream_threads(WQ);
  constexpr int SUB = C::SUB, S = C::S, WK = kSWarps / WQ, NT = kSKeys / 8, KS = HD / 16, OLD = C::OLD;
  constexpr int ROWS = WQ * 16;
  static_assert(S % WK == 0, "each group owns its stages");
  static_assert(kSWarps * 16 * OLD * 4 <= S * (int)C::kTile, "partial outputs fit over the ring");

  extern __shared__ unsigned char smem_raw[];
  __shared__ __align__(8) unsigned long long full_bar[S], empty_bar[S];
  __shared__ int issued_s;                         // tiles that the producer requested
  __shared__ float2 ml[kSWarps][16];              // (max, sum) per warp and query row
  __shared__ __align__(8) float2 ml_cta[ROWS];    // after the merge of the CTA's key groups

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g4 = lane >> 2, t4 = lane & 3;
  const int split = blockIdx.x, ns = gridDim.x;
  const int group = a.hq / a.hkv;
  int b, row0, nrows;
  seg_of(a.segs, blockIdx.z, b, row0, nrows);
  const int kvh = blockIdx.y % a.hkv;
  const int nq = group * nrows;                   // queries of this kv head, row-major: q = j * group + g
  const int nqg = (nq + ROWS - 1) / ROWS;
  const int qi = blockIdx.y / a.hkv;
  if (qi >= nqg) return;                          // a shorter segment (the same for every split of the cluster)
  const int qg = nqg - 1 - qi;                    // the groups that see most keys start first
  const int qd = a.hq * HD;

  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  float *obuf = reinterpret_cast<float *>(smem_raw + (base - smem_u32(smem_raw)));     // [4 warps][16][OLD], over the ring

  const int L = a.kv_len[b];
  const int q_first = qg * ROWS;
  const int q_last = min(nq, q_first + ROWS) - 1;
  const int n_all = (L + q_last / group + kSKeys) / kSKeys;           // tiles up to the last visible key L + j
  const int tps = (n_all + ns - 1) / ns;
  const int t_begin = min(n_all, split * tps);
  const int nt = min(n_all, t_begin + tps) - t_begin;

  if (tid == 0) {
    for (int i = 0; i < S; ++i) { mbar_init(smem_u32(&full_bar[i]), 1); mbar_init(smem_u32(&empty_bar[i]), WQ); }
    fence_barrier_init();
    fence_proxy_async();
  }
  __syncthreads();
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

  bool ok = true;
  float m_run[2] = {-INFINITY, -INFINITY}, l_run[2] = {0.f, 0.f}, o[HD / 8][4];
#pragma unroll
  for (int n = 0; n < HD / 8; ++n)
#pragma unroll
    for (int i = 0; i < 4; ++i) o[n][i] = 0.f;
  const int wq = warp % WQ, kg = warp / WQ;

  if (warp == kSWarps) {
    // ---- producer: tiles of keys that earlier steps wrote are requested before the kernel in front has finished
    if (lane == 0) {
      const int plane_k = a.k_plane0 + b * a.hkv + kvh, plane_v = a.v_plane0 + b * a.hkv + kvh;
      bool waited = false;
      int t = 0;
      for (; t < nt; ++t) {
        const int stage = t % S;
        if (t >= S && !wait_bounded(smem_u32(&empty_bar[stage]), (uint32_t)(t / S - 1) & 1u)) { ok = false; break; }
        const int y = (t_begin + t) * kSKeys;
        if (!waited && y + kSKeys > L) {
          asm volatile("griddepcontrol.wait;" ::: "memory");
          asm volatile("fence.proxy.async;" ::: "memory");       // rows stored by the kernel in front, read by the TMA
          waited = true;
        }
        const uint32_t bar = smem_u32(&full_bar[stage]), dst = base + stage * C::kTile;
        mbar_expect_tx(bar, C::kTile);
#pragma unroll
        for (int s = 0; s < SUB; ++s) load_3d(dst + s * C::kSub, &map, s * 64, y, plane_k, bar);
#pragma unroll
        for (int s = 0; s < SUB; ++s) load_3d(dst + C::kHalf + s * C::kSub, &map, s * 64, y, plane_v, bar);
      }
      issued_s = t;
    }
  } else {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    // ---- this warp's 16 query rows as MMA A fragments (rows beyond the last query hold anything; nothing is stored for them)
    uint32_t qh[KS][4], ql[KS][4];
    {
      const int tile = min(seg_tile0(row0, group, blockIdx.z) + qg * WQ + wq, a.q_tiles - 1);      // a tile beyond the segment's is never stored
      const uint4 *p = (const uint4 *)a.q + q_frag(kvh, a.q_tiles, tile, 0, 0, HD) * 32 + lane;
#pragma unroll
      for (int ks = 0; ks < KS; ++ks) {
        const uint4 h = __ldcg(p + ks * 32), w = __ldcg(p + (KS + ks) * 32);
        qh[ks][0] = h.x; qh[ks][1] = h.y; qh[ks][2] = h.z; qh[ks][3] = h.w;
        ql[ks][0] = w.x; ql[ks][1] = w.y; ql[ks][2] = w.z; ql[ks][3] = w.w;
      }
    }
    int lim[2];                                                   // last visible key of rows g4 and g4 + 8
#pragma unroll
    for (int hh = 0; hh < 2; ++hh) lim[hh] = L + min(q_first + wq * 16 + g4 + hh * 8, nq - 1) / group;
    const int q_hi = min(nq - 1, q_first + wq * 16 + 15), q_lo = min(nq - 1, q_first + wq * 16);
    const int warp_last = L + q_hi / group, warp_first = L + q_lo / group;     // last visible key of the warp's last / first row
    const int last_key = L + nrows - 1;                           // beyond it the slab holds anything
    const float sl2 = rsqrtf((float)HD) * 1.4426950408889634f;

    for (int t = kg; t < nt; t += WK) {
      const int stage = t % S, key0 = (t_begin + t) * kSKeys;
      // the verdict is made uniform: lanes that leave the poll at different times must be one warp again before the
      // warp-wide matrix instructions
      if (!__all_sync(0xffffffffu, wait_bounded(smem_u32(&full_bar[stage]), (uint32_t)(t / S) & 1u))) { ok = false; break; }
      if (key0 <= warp_last) {
        const uint32_t kb = base + stage * C::kTile, vb = kb + C::kHalf;
        if (key0 + kSKeys - 1 > last_key) {
          // values beyond the last written key: a zero probability would still multiply a NaN pattern.  (The warps of
          // a tile write the same zeros; no tile follows this one in its stage.)
          unsigned char *vg = smem_raw + (vb - smem_u32(smem_raw));
          for (int e = lane; e < (key0 + kSKeys - 1 - last_key) * (HD / 8); e += 32) {
            const int row = last_key + 1 - key0 + e / (HD / 8), ch = e % (HD / 8);
            *reinterpret_cast<uint4 *>(vg + soff(row, ch)) = make_uint4(0, 0, 0, 0);
          }
          __syncwarp();
        }
        // ---- S = Q.K^T: 16 rows x 32 keys
        float s[NT][4];
#pragma unroll
        for (int n = 0; n < NT; ++n)
#pragma unroll
          for (int i = 0; i < 4; ++i) s[n][i] = 0.f;
#pragma unroll
        for (int k2 = 0; k2 < KS / 2; ++k2) {
          uint32_t kf[NT][4];
#pragma unroll
          for (int n = 0; n < NT; ++n) ldsm4(kb + soff(n * 8 + (lane & 7), k2 * 4 + (lane >> 3)), kf[n]);
#pragma unroll
          for (int n = 0; n < NT; ++n) mma16816(s[n], qh[2 * k2], kf[n][0], kf[n][1]);
#pragma unroll
          for (int n = 0; n < NT; ++n) mma16816(s[n], ql[2 * k2], kf[n][0], kf[n][1]);
#pragma unroll
          for (int n = 0; n < NT; ++n) mma16816(s[n], qh[2 * k2 + 1], kf[n][2], kf[n][3]);
#pragma unroll
          for (int n = 0; n < NT; ++n) mma16816(s[n], ql[2 * k2 + 1], kf[n][2], kf[n][3]);
        }
        // ---- causal mask (tiles that reach beyond the first row's last key only), running maximum
        if (key0 + kSKeys - 1 > warp_first) {
#pragma unroll
          for (int n = 0; n < NT; ++n)
#pragma unroll
            for (int i = 0; i < 4; ++i)
              if (key0 + n * 8 + t4 * 2 + (i & 1) > lim[i >> 1]) s[n][i] = -INFINITY;
        }
        float mx[2] = {m_run[0], m_run[1]};
#pragma unroll
        for (int n = 0; n < NT; ++n) {
          mx[0] = fmaxf(mx[0], fmaxf(s[n][0], s[n][1]));
          mx[1] = fmaxf(mx[1], fmaxf(s[n][2], s[n][3]));
        }
#pragma unroll
        for (int hh = 0; hh < 2; ++hh) {
          mx[hh] = fmaxf(mx[hh], __shfl_xor_sync(0xffffffffu, mx[hh], 1));
          mx[hh] = fmaxf(mx[hh], __shfl_xor_sync(0xffffffffu, mx[hh], 2));
        }
        if (__any_sync(0xffffffffu, mx[0] > m_run[0] || mx[1] > m_run[1])) {
          float corr[2];
#pragma unroll
          for (int hh = 0; hh < 2; ++hh) {
            corr[hh] = mx[hh] == -INFINITY ? 1.f : ex2((m_run[hh] - mx[hh]) * sl2);     // first tile: 2^-inf = 0
            l_run[hh] *= corr[hh];
            m_run[hh] = mx[hh];
          }
#pragma unroll
          for (int n = 0; n < HD / 8; ++n) { o[n][0] *= corr[0]; o[n][1] *= corr[0]; o[n][2] *= corr[1]; o[n][3] *= corr[1]; }
        }
        // ---- probabilities; P.V with the score registers as the A operand
        const float mb[2] = {m_run[0] == -INFINITY ? 0.f : m_run[0] * sl2, m_run[1] == -INFINITY ? 0.f : m_run[1] * sl2};
#pragma unroll
        for (int n = 0; n < NT; ++n) {
#pragma unroll
          for (int i = 0; i < 4; ++i) s[n][i] = ex2(fmaf(s[n][i], sl2, -mb[i >> 1]));
          l_run[0] += s[n][0] + s[n][1];
          l_run[1] += s[n][2] + s[n][3];
        }
#pragma unroll
        for (int kk = 0; kk < NT / 2; ++kk) {
          uint32_t ph[4], pl[4];
#pragma unroll
          for (int x = 0; x < 4; ++x) {
            const float p0 = s[2 * kk + (x >> 1)][(x & 1) * 2], p1 = s[2 * kk + (x >> 1)][(x & 1) * 2 + 1];
            ph[x] = pack2(p0, p1);
            pl[x] = pack2(p0 - low_half(ph[x]), p1 - high_half(ph[x]));
          }
#pragma unroll
          for (int n4 = 0; n4 < HD / 32; ++n4) {
            uint32_t vf[2][4];
            ldsm4t(vb + soff(kk * 16 + (lane & 15), n4 * 4 + (lane >> 4)), vf[0]);
            ldsm4t(vb + soff(kk * 16 + (lane & 15), n4 * 4 + 2 + (lane >> 4)), vf[1]);
#pragma unroll
            for (int x = 0; x < 4; ++x) mma16816(o[4 * n4 + x], ph, vf[x >> 1][(x & 1) * 2], vf[x >> 1][(x & 1) * 2 + 1]);
#pragma unroll
            for (int x = 0; x < 4; ++x) mma16816(o[4 * n4 + x], pl, vf[x >> 1][(x & 1) * 2], vf[x >> 1][(x & 1) * 2 + 1]);
          }
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&empty_bar[stage]));
    }
#pragma unroll
    for (int hh = 0; hh < 2; ++hh) {
      l_run[hh] += __shfl_xor_sync(0xffffffffu, l_run[hh], 1);
      l_run[hh] += __shfl_xor_sync(0xffffffffu, l_run[hh], 2);
    }
  }
  if (!__syncthreads_and(ok ? 1 : 0)) {
    // a tile did not arrive: no result.  Copies on their way are waited for (bounded).
    if (tid == 0) {
      atomicExch(a.err, 1u);
      const unsigned long long t0 = clock64();
      for (int i = 0; i < S && i < issued_s; ++i)
        while (!mbar_try(smem_u32(&full_bar[i]), last_copy_parity(issued_s, S, i)))
          if ((unsigned long long)(clock64() - t0) > kSpinBudget / 4) break;
    }
    __syncthreads();
  }

  // ---- partial results of the warps
  if (warp < kSWarps) {
    float *ob = obuf + warp * 16 * OLD;
#pragma unroll
    for (int n = 0; n < HD / 8; ++n) {
      *reinterpret_cast<float2 *>(ob + g4 * OLD + n * 8 + t4 * 2) = make_float2(o[n][0], o[n][1]);
      *reinterpret_cast<float2 *>(ob + (g4 + 8) * OLD + n * 8 + t4 * 2) = make_float2(o[n][2], o[n][3]);
    }
    if (t4 == 0) { ml[warp][g4] = make_float2(m_run[0], l_run[0]); ml[warp][g4 + 8] = make_float2(m_run[1], l_run[1]); }
  }
  __syncthreads();
  const float sl2 = rsqrtf((float)HD) * 1.4426950408889634f;
  auto store = [&](int row, int c4, float4 v) {
    const int q = q_first + row;
    const int j = q / group, h = kvh * group + q - j * group;
    const long long at = (long long)(row0 + j) * qd + h * HD + c4 * 4;
    if (a.out_pan) {
      const uint2 hi = make_uint2(pack2(v.x, v.y), pack2(v.z, v.w));
      __nv_bfloat16 *p = (__nv_bfloat16 *)a.out_pan + at;
      *reinterpret_cast<uint2 *>(p) = hi;
      *reinterpret_cast<uint2 *>(p + (long long)a.pan_rows * qd) =
          make_uint2(pack2(v.x - low_half(hi.x), v.y - high_half(hi.x)), pack2(v.z - low_half(hi.y), v.w - high_half(hi.y)));
    } else {
      *reinterpret_cast<float4 *>(a.out + at) = v;
    }
  };
  // ---- merge of the CTA's key groups; with one split this is the result
  for (int u = tid; u < ROWS * (HD / 4); u += kSThreads) {
    const int row = u / (HD / 4), c4 = u - row * (HD / 4);
    const int w0 = row >> 4, rr = row & 15;
    float M = -INFINITY;
#pragma unroll
    for (int k = 0; k < WK; ++k) M = fmaxf(M, ml[k * WQ + w0][rr].x);
    float den = 0.f;
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int k = 0; k < WK; ++k) {
      const float2 v = ml[k * WQ + w0][rr];
      const float w = v.x == -INFINITY ? 0.f : ex2((v.x - M) * sl2);
      const float4 x = *reinterpret_cast<const float4 *>(obuf + ((k * WQ + w0) * 16 + rr) * OLD + c4 * 4);
      den = fmaf(v.y, w, den);
      acc.x = fmaf(w, x.x, acc.x); acc.y = fmaf(w, x.y, acc.y); acc.z = fmaf(w, x.z, acc.z); acc.w = fmaf(w, x.w, acc.w);
    }
    if (ns == 1) {
      if (q_first + row < nq) {
        const float inv = 1.0f / den;
        store(row, c4, make_float4(acc.x * inv, acc.y * inv, acc.z * inv, acc.w * inv));
      }
    } else {
      *reinterpret_cast<float4 *>(obuf + (w0 * 16 + rr) * OLD + c4 * 4) = acc;          // only this thread reads these
      if (c4 == 0) ml_cta[row] = make_float2(M, den);
    }
  }
  if (ns == 1) return;
  // ---- merge of the key splits through the cluster's shared memory
  cluster_sync_all();
  const uint32_t ml_addr = smem_u32(ml_cta);
  for (int u = split * kSThreads + tid; u < ROWS * (HD / 4); u += ns * kSThreads) {
    const int row = u / (HD / 4), c4 = u - row * (HD / 4);
    if (q_first + row >= nq) continue;
    float2 mv[8];
    float4 ov[8];
#pragma unroll
    for (int sp = 0; sp < 8; ++sp) {
      mv[sp] = make_float2(-INFINITY, 0.f);
      ov[sp] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (sp < ns) {
        mv[sp] = ld_cluster_f2(map_to_cta(ml_addr + (uint32_t)row * 8u, (uint32_t)sp));
        ov[sp] = ld_cluster_f4(map_to_cta(base + (uint32_t)(row * OLD + c4 * 4) * 4u, (uint32_t)sp));
      }
    }
    float M = -INFINITY;
#pragma unroll
    for (int sp = 0; sp < 8; ++sp) M = fmaxf(M, mv[sp].x);
    float den = 0.f;
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int sp = 0; sp < 8; ++sp) {
      const float w = mv[sp].x == -INFINITY ? 0.f : ex2((mv[sp].x - M) * sl2);
      den = fmaf(mv[sp].y, w, den);
      acc.x = fmaf(w, ov[sp].x, acc.x); acc.y = fmaf(w, ov[sp].y, acc.y);
      acc.z = fmaf(w, ov[sp].z, acc.z); acc.w = fmaf(w, ov[sp].w, acc.w);
    }
    const float inv = 1.0f / den;
    store(row, c4, make_float4(acc.x * inv, acc.y * inv, acc.z * inv, acc.w * inv));
  }
  cluster_sync_all();                                            // the other splits may still be reading this CTA's memory
}

// ------------------------------------------------------------------------------------ host side
cudaError_t launch_qkv_finish(const QkvFinishArgs &a, int R, cudaStream_t st) {
  if (R < 1 || a.hd % 8 || (a.segs.n == 0 && a.segs.c < 1) || a.segs.n > kMaxSegs) return cudaErrorInvalidValue;
  const int units = (a.hq + 2 * a.hkv) * (a.hd >> 3);
  int ny = (4 * 148 + R - 1) / R;                   // about four blocks per SM when there are few rows
  if (ny > (units + 255) / 256) ny = (units + 255) / 256;
  cudaLaunchConfig_t cfg;
  memset(&cfg, 0, sizeof cfg);
  cfg.gridDim = dim3(R, ny); cfg.blockDim = dim3(256); cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr; cfg.numAttrs = a.pdl ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, qkv_finish_kernel, a);
}

template <int HD, int WQ>
static cudaError_t stream_config(cudaLaunchConfig_t &cfg, cudaLaunchAttribute (&attr)[2], int ns, int ny, int nz, bool pdl, cudaStream_t st) {
  const size_t smem = StreamCfg<HD>::smem();
  static bool attr_done[kMaxDevices] = {false};
  const int dev = current_device_slot();
  if (!attr_done[dev]) {
    cudaError_t e = cudaFuncSetAttribute(attn_stream_kernel<HD, WQ>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    attr_done[dev] = true;
  }
  memset(&cfg, 0, sizeof cfg);
  cfg.gridDim = dim3(ns, ny, nz); cfg.blockDim = dim3(stream_threads(WQ)); cfg.dynamicSmemBytes = smem; cfg.stream = st;
  int na = 0;
  if (pdl) {
    attr[na].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[na].val.programmaticStreamSerializationAllowed = 1;
    ++na;
  }
  if (ns > 1) {
    attr[na].id = cudaLaunchAttributeClusterDimension;
    attr[na].val.clusterDim.x = (unsigned)ns; attr[na].val.clusterDim.y = 1; attr[na].val.clusterDim.z = 1;
    ++na;
  }
  cfg.attrs = attr; cfg.numAttrs = na;
  return cudaSuccess;
}

// Clusters of ns CTAs that run at the same time.  Clusters do not cross groups of SMs, so it is fewer than CTA slots / ns (B200:
// 296 slots, 71 clusters of four, 45 of six, 37 of seven, 33 of eight); a sixteenth is left out, because the CTAs of the kernel in
// front still hold slots when they are placed (32 clusters of eight ran in two rounds).
template <int HD, int WQ>
static int stream_clusters_t(int ns, int n_sms) {
  if (ns == 1) return 2 * n_sms;
  static int known[kMaxDevices][9] = {};
  int &n = known[current_device_slot()][ns];
  if (n == 0) {
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[2];
    int fit = 0;
    if (stream_config<HD, WQ>(cfg, attr, ns, 1, 1, false, nullptr) != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&fit, attn_stream_kernel<HD, WQ>, &cfg) != cudaSuccess || fit < 1) {
      (void)cudaGetLastError();
      fit = 1;
    }
    n = fit > 15 ? fit * 15 / 16 : fit;
  }
  return n;
}
static int stream_clusters(int hd, int wq, int ns, int n_sms) {
  if (hd == 128) return wq == 1 ? stream_clusters_t<128, 1>(ns, n_sms) : wq == 2 ? stream_clusters_t<128, 2>(ns, n_sms) : stream_clusters_t<128, 4>(ns, n_sms);
  return wq == 1 ? stream_clusters_t<64, 1>(ns, n_sms) : wq == 2 ? stream_clusters_t<64, 2>(ns, n_sms) : stream_clusters_t<64, 4>(ns, n_sms);
}

// Query tiles per CTA and key splits for `nb` segments of at most `rows` rows behind at most max_len keys.
static void stream_plan(int max_len, int rows, int group, int hkv, int nb, int hd, int n_sms, bool spare, int &wq, int &ns) {
  const int nqt = (group * rows + 15) / 16;
  wq = nqt >= 3 ? 4 : nqt;
  const long long units = (long long)nb * hkv * ((nqt + wq - 1) / wq);
  const int tiles = (max_len + rows + kSKeys - 1) / kSKeys;
  // Rounds of clusters times a CTA's length in tile times; start, query loads and merge cost about as much as six tiles.  Measured
  // by splits, 4 layers over 8000 keys: 7B, 1 x 32 rows (32 units) 4 splits 825 us, 6 742, 7 720, 8 822; 13B, 1 x 32 (40 units) 5
  // 931, 6 894, 7 1028; 13B, 2 x 16 (80 units) 2 957, 3 914, 4 1002; 7B, 4 x 16 (128 units) 1 1084, 2 940, 3 1003.
  // Behind a persistent launch of projections, where clusters that only just fit run in two rounds (spare): one-writer, 1.1B, 13 x 4 rows over 5000 keys
  // (52 clusters of five) 2176 -> 1988 us a step, 26 heads of 128 (268 MB, 6 layers), 2 x 32 over 8000
  // 1235 -> 1128; chained, 2 x 40 over 2000 1039 -> 1010, over 8000 1610 -> 1551; 34 clusters of seven, 1 x 64 over 8000 992 -> 965.  Behind the dense
  // GEMMs, whose clusters leave one by one, it only takes splits away: 22 heads, 3 x 48 over 4000 891 -> 973, 34 heads, 4 x 40 1496 -> 1668 (4 layers).
  // (With two rounds or more the edge does not show: 1.1B, 13 x 16 over 4000 3626 -> 3793.)
  ns = stream_splits(tiles, units, spare, [&](int s) { return stream_clusters(hd, wq, s, n_sms); });
}

template <int HD, int WQ>
static cudaError_t launch_stream_t(const KvTensorMap &map, const StreamAttnArgs &a, int ns, int nqg, int nseg, cudaStream_t st) {
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr[2];
  cudaError_t e = stream_config<HD, WQ>(cfg, attr, ns, a.hkv * nqg, nseg, a.pdl != 0, st);
  return e == cudaSuccess ? cudaLaunchKernelEx(&cfg, attn_stream_kernel<HD, WQ>, *reinterpret_cast<const CUtensorMap *>(&map), a) : e;
}

cudaError_t launch_attn_stream(const KvTensorMap &map, const StreamAttnArgs &a, int nseg, int max_rows, int max_len, int hd,
                               int n_sms, cudaStream_t st) {
  if (nseg < 1 || nseg > 65535 || max_rows < 1 || !a.err || a.segs.n > kMaxSegs || (hd != 64 && hd != 128)) return cudaErrorInvalidValue;
  const int group = a.hq / a.hkv;
  int wq, ns;
  stream_plan(max_len, max_rows, group, a.hkv, nseg, hd, n_sms, a.spare != 0, wq, ns);
  const int nqg = (group * max_rows + wq * 16 - 1) / (wq * 16);
  if ((long long)a.hkv * nqg > 65535) return cudaErrorInvalidValue;
  if (hd == 128) {
    if (wq == 1) return launch_stream_t<128, 1>(map, a, ns, nqg, nseg, st);
    if (wq == 2) return launch_stream_t<128, 2>(map, a, ns, nqg, nseg, st);
    return launch_stream_t<128, 4>(map, a, ns, nqg, nseg, st);
  }
  if (wq == 1) return launch_stream_t<64, 1>(map, a, ns, nqg, nseg, st);
  if (wq == 2) return launch_stream_t<64, 2>(map, a, ns, nqg, nseg, st);
  return launch_stream_t<64, 4>(map, a, ns, nqg, nseg, st);
}

// Where this pair of kernels is faster than the fused one (attn_tma_kernel): with at least 64 units (kv head of a sequence x
// 16 queries) that read together at least a thousand tiles of 64 keys, three or more each.  Measured, time of an 8-layer step,
// fused -> this: 7B, 16 x 1 row, 512 keys 1107 -> 1048 us, 16 x 4 rows, 1024 keys 1608 -> 1470; 4 x 16 rows, 512 keys 1220 -> 1176;
// 1.1B, 16 x 1, 1024 keys 508 -> 473, 16 x 16, 512 keys 1331 -> 1210; 13B, 8 x 32, 2048 keys 4600 -> 4230; of a 4-layer step over
// 8000 keys: 7B, 1 x 32 778 -> 720, 13B, 1 x 32 998 -> 894.  Below the line the second launch per layer costs about what it brings
// or more: 7B, 2 x 8, 512 keys 882 -> 894; 1.1B, 4 x 4, 1024 keys 469 -> 476, and over two tiles of keys (64 keys; 4 layers)
// 7B, 16 x 1 499 -> 535, 16 x 4 665 -> 664 to 744, 13B, 16 x 1 678 -> 678.
bool attn_stream_pays(int max_len, int c, int hq, int hkv, int nb) {
  const long long units = (long long)nb * hkv * (((long long)(hq / hkv) * c + 15) / 16);
  const int tiles = (max_len + c + 63) / 64;
  return units >= 64 && tiles >= 3 && units * tiles >= 1000;
}

int attn_stream_tile_keys() { return kSKeys; }
size_t attn_stream_q_tiles(int rows, int group, int nseg) { return (size_t)rows * group / 16 + nseg + 1; }

}  // namespace fc
