// Window attention of few (sequence, kv head, 16-query) units over short caches, with everything around it in the same
// kernel: 1/rms and rotation of the queries and of the window's keys out of the fp32 QKV accumulators, K/V rows into the cache.
//
// What bounds it: latency from the QKV projection's end to the output projection's operand - the K/V bytes (13 MB per layer of
// 7B over 800 keys) are on their way before the kernel in front has finished.  So the chain behind that point is
// kept short: grid (key splits, kv heads x query tiles, sequences), the splits of a unit are one cluster; four warps,
// each on 32-key tiles of its own (its own ring stages, requested by itself: no producer, no block-wide barrier per tile), queries in
// the registers of MMA A operands, scores and output in registers (the accumulators of Q.K^T are the A operand of P.V as they are), one merge of the warps and one of the splits.  The last split also turns the
// window's own keys and values into bf16 in shared memory and in the cache; blocks of 16 window keys are causal.
// q and the probabilities enter the tensor cores as bf16 pairs, so that only the stored K/V are rounded.
// Row j of a sequence sees keys 0 .. kv_len + j.  Every wait is bounded.
#include <cstring>

#include "fc_attn.cuh"
#include "fc_internal.h"
#include "fc_plan.h"
#include "fc_ptx.cuh"

namespace fc {

namespace {
constexpr int kShortKeys = 32;                     // keys per tile
constexpr int kShortWarps = 4, kShortThreads = kShortWarps * 32;
constexpr int kShortStages = 4;                    // tiles in flight per warp at most

template <int HD>
struct ShortCfg {
  static constexpr int SUB = HD / 64;              // 128-byte sub-tiles per row
  static constexpr uint32_t kSub = kShortKeys * 128;
  static constexpr uint32_t kHalf = SUB * kSub;    // K (or V) of a tile
  static constexpr uint32_t kTile = 2 * kHalf;     // 16 KB, 8 KB
  static constexpr uint32_t kQ = 16 * HD * 4;      // 16 queries, high and low
  static constexpr int stages(bool deep) { return (deep ? 2 : 1) * (HD == 64 ? 2 : 1); }      // tiles in flight per warp
  static constexpr int OLD = HD + 8;               // row pitch of the partial outputs (floats): spreads the banks
  static_assert(kShortWarps * 16 * OLD * 4 <= kShortWarps * (int)kTile, "partial outputs fit over one stage per warp");
};
template <int HD> size_t short_smem(int c, int stages) {
  return 1024 + (size_t)kShortWarps * stages * ShortCfg<HD>::kTile + (size_t)((c + 15) / 16 * 16) * HD * 4 + ShortCfg<HD>::kQ;
}

// Byte offset of 16-byte piece `ch` of row `r` in sub-tiles of 128-byte rows, `sub` bytes apart, with the TMA's swizzle.
__device__ __forceinline__ uint32_t piece(int r, int ch, uint32_t sub) {
  return (uint32_t)(ch >> 3) * sub + (uint32_t)r * 128u + (uint32_t)(((ch & 7) ^ (r & 7)) << 4);
}

// One block of 8 * NT keys: scores, probabilities, output of a warp's 16 queries.  vis(n, i): key 8 n + 2 (lane & 3) + (i & 1) is
// visible to the row of accumulator i; all: every key is to every row.
template <int HD, int NT, typename Vis>
__device__ __forceinline__ void attend(uint32_t kb, uint32_t vb, uint32_t sub, const uint32_t (&qh)[HD / 16][4], const uint32_t (&ql)[HD / 16][4],
                                       float (&o)[HD / 8][4], float (&m_run)[2], float (&l_run)[2], float sl2, int lane, bool all, Vis vis) {
  float s[NT][4];
#pragma unroll
  for (int n = 0; n < NT; ++n)
#pragma unroll
    for (int i = 0; i < 4; ++i) s[n][i] = 0.f;
#pragma unroll
  for (int k2 = 0; k2 < HD / 32; ++k2) {
    uint32_t kf[NT][4];
#pragma unroll
    for (int n = 0; n < NT; ++n) ldsm4(kb + piece(n * 8 + (lane & 7), k2 * 4 + (lane >> 3), sub), kf[n]);
#pragma unroll
    for (int n = 0; n < NT; ++n) mma16816(s[n], qh[2 * k2], kf[n][0], kf[n][1]);
#pragma unroll
    for (int n = 0; n < NT; ++n) mma16816(s[n], ql[2 * k2], kf[n][0], kf[n][1]);
#pragma unroll
    for (int n = 0; n < NT; ++n) mma16816(s[n], qh[2 * k2 + 1], kf[n][2], kf[n][3]);
#pragma unroll
    for (int n = 0; n < NT; ++n) mma16816(s[n], ql[2 * k2 + 1], kf[n][2], kf[n][3]);
  }
  if (!all) {
#pragma unroll
    for (int n = 0; n < NT; ++n)
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (!vis(n, i)) s[n][i] = -INFINITY;
  }
  float mx[2] = {m_run[0], m_run[1]};
#pragma unroll
  for (int n = 0; n < NT; ++n) {
    mx[0] = fmaxf(mx[0], fmaxf(s[n][0], s[n][1]));
    mx[1] = fmaxf(mx[1], fmaxf(s[n][2], s[n][3]));
  }
  float mb[2];
#pragma unroll
  for (int hh = 0; hh < 2; ++hh) {
    mx[hh] = fmaxf(mx[hh], __shfl_xor_sync(0xffffffffu, mx[hh], 1));
    mx[hh] = fmaxf(mx[hh], __shfl_xor_sync(0xffffffffu, mx[hh], 2));
    const float corr = mx[hh] == -INFINITY ? 1.f : ex2((m_run[hh] - mx[hh]) * sl2);       // first block: 2^-inf = 0
    l_run[hh] *= corr;
    m_run[hh] = mx[hh];
    mb[hh] = mx[hh] == -INFINITY ? 0.f : mx[hh] * sl2;
#pragma unroll
    for (int n = 0; n < HD / 8; ++n) { o[n][2 * hh] *= corr; o[n][2 * hh + 1] *= corr; }
  }
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
      ldsm4t(vb + piece(kk * 16 + (lane & 15), n4 * 4 + (lane >> 4), sub), vf[0]);
      ldsm4t(vb + piece(kk * 16 + (lane & 15), n4 * 4 + 2 + (lane >> 4), sub), vf[1]);
#pragma unroll
      for (int x = 0; x < 4; ++x) mma16816(o[4 * n4 + x], ph, vf[x >> 1][(x & 1) * 2], vf[x >> 1][(x & 1) * 2 + 1]);
#pragma unroll
      for (int x = 0; x < 4; ++x) mma16816(o[4 * n4 + x], pl, vf[x >> 1][(x & 1) * 2], vf[x >> 1][(x & 1) * 2 + 1]);
    }
  }
}
}  // namespace

template <int HD>
__global__ void __launch_bounds__(kShortThreads, 2)
attn_short_kernel(const __grid_constant__ CUtensorMap map, const __grid_constant__ ShortAttnArgs a) {
  using C = ShortCfg<HD>;
  constexpr int HALF = HD / 2, KS = HD / 16, OLD = C::OLD;
  extern __shared__ unsigned char smem_raw[];
  __shared__ __align__(8) unsigned long long full_bar[kShortWarps][kShortStages];
  __shared__ float2 ml[kShortWarps][16];           // (max, sum) per warp and query row
  __shared__ __align__(8) float2 ml_cta[16];       // after the merge of the CTA's warps
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g4 = lane >> 2, t4 = lane & 3;
  const int split = blockIdx.x, ns = gridDim.x, NS = a.stages;
  const int group = a.hq / a.hkv, c = a.c, nq = group * c;
  const int kvh = blockIdx.y % a.hkv, q0 = (blockIdx.y / a.hkv) * 16;                 // first query of the tile; query q = row * group + head of the group
  const int bl = blockIdx.z, b = a.seq_map ? a.seq_map[bl] : a.b0 + bl;
  const int qd = a.hq * HD, kvd = a.hkv * HD;
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  unsigned char *gen = smem_raw + (base - smem_u32(smem_raw));
  float *obuf = reinterpret_cast<float *>(gen);    // [warps][16][OLD], over the ring
  const int wrows = (c + 15) & ~15;
  const uint32_t wsub = (uint32_t)wrows * 128u, win_k = base + (uint32_t)(kShortWarps * NS) * C::kTile, win_v = win_k + C::SUB * wsub;
  unsigned char *q_area = gen + (win_v - base) + C::SUB * wsub;

  const int L = a.kv_len[b];
  const int n_all = (L + kShortKeys - 1) / kShortKeys;                               // tiles of cached keys
  const int n_cta = n_all > split ? (n_all - split + ns - 1) / ns : 0;               // this CTA's: split, split + ns, ...
  const int n_mine = n_cta > warp ? (n_cta - warp + kShortWarps - 1) / kShortWarps : 0;       // this warp's: every fourth of them
  const int plane_k = a.k_plane0 + b * a.hkv + kvh, plane_v = a.v_plane0 + b * a.hkv + kvh;
  const uint32_t ring = base + (uint32_t)(warp * NS) * C::kTile;
  auto key0_of = [&](int i) { return (split + (warp + i * kShortWarps) * ns) * kShortKeys; };
  auto request = [&](int i) {                      // lane 0
    const int stage = i % NS;
    const uint32_t bar = smem_u32(&full_bar[warp][stage]), dst = ring + (uint32_t)stage * C::kTile;
    const int y = key0_of(i);
    mbar_expect_tx(bar, C::kTile);
#pragma unroll
    for (int s = 0; s < C::SUB; ++s) load_3d(dst + s * C::kSub, &map, s * 64, y, plane_k, bar);
#pragma unroll
    for (int s = 0; s < C::SUB; ++s) load_3d(dst + C::kHalf + s * C::kSub, &map, s * 64, y, plane_v, bar);
  };
  if (lane == 0) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(&map) : "memory");
    for (int i = 0; i < kShortStages; ++i) mbar_init(smem_u32(&full_bar[warp][i]), 1);
    fence_barrier_init();
    fence_proxy_async();
    // cached keys were written by earlier steps
    for (int i = 0; i < NS && i < n_mine; ++i) request(i);
  }
  __syncwarp();
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");

  // Queries and window keys by loops of few instructions over the block: code that runs once per launch costs its fetch (each warp
  // straight from the accumulators into its registers, 128 loads unrolled: 4 us).
  // ---- queries, in the order in which a warp holds them as MMA A operands: [high, low][16-wide k block][lane][4 registers]
  {
    constexpr int PT = HALF / 8;                   // pairs (i, i + HALF) per thread: 8 or 4 adjacent ones
    const int rr = tid >> 3, q = q0 + rr;
    const bool live = q < nq;
    const int j = live ? q / group : 0, r = bl * c + j, i0 = (tid & 7) * PT;
    const float *src = a.qkv + (long long)r * a.ldq + (kvh * group + (live ? q - j * group : 0)) * HD + i0;
    const float4 *rot = reinterpret_cast<const float4 *>(a.rope + (long long)(L + j) * HALF + i0);
    float4 u[PT / 4], w[PT / 4], t[PT / 2];
    const float ss = __ldcg(a.ss + r);
#pragma unroll
    for (int k = 0; k < PT / 4; ++k) { u[k] = __ldcg(reinterpret_cast<const float4 *>(src) + k); w[k] = __ldcg(reinterpret_cast<const float4 *>(src + HALF) + k); }
#pragma unroll
    for (int k = 0; k < PT / 2; ++k) t[k] = __ldg(rot + k);
    const float s = live ? rsqrtf(ss / (float)a.dn + a.eps) : 0.f;
    uint32_t *qs = reinterpret_cast<uint32_t *>(q_area);
#pragma unroll
    for (int k = 0; k < PT / 2; ++k) {             // two adjacent pairs: one register of the low, one of the high half of the head
      const float u0 = ((k & 1) ? u[k >> 1].z : u[k >> 1].x) * s, u1 = ((k & 1) ? u[k >> 1].w : u[k >> 1].y) * s;
      const float w0 = ((k & 1) ? w[k >> 1].z : w[k >> 1].x) * s, w1 = ((k & 1) ? w[k >> 1].w : w[k >> 1].y) * s;
      const float a0 = u0 * t[k].x - w0 * t[k].y, a1 = u1 * t[k].z - w1 * t[k].w, b0 = u0 * t[k].y + w0 * t[k].x, b1 = u1 * t[k].w + w1 * t[k].z;
      const int e = i0 + 2 * k, at = ((e >> 4) * 32 + (rr & 7) * 4 + ((e & 7) >> 1)) * 4 + (rr >> 3) + 2 * ((e & 15) >> 3);
      const uint32_t h0 = pack2(a0, a1), h1 = pack2(b0, b1);
      qs[at] = h0; qs[at + (KS / 2) * 128] = h1;
      qs[at + KS * 128] = pack2(a0 - low_half(h0), a1 - high_half(h0));
      qs[at + (KS + KS / 2) * 128] = pack2(b0 - low_half(h1), b1 - high_half(h1));
    }
  }
  // ---- the window's own keys and values (last split)
  const bool has_win = split == ns - 1;
  if (has_win) {
    const bool store = q0 == 0;                    // one query tile of the kv head writes the cache
    __nv_bfloat16 *kc = (__nv_bfloat16 *)a.kcache + (long long)b * a.stride_b + (long long)kvh * a.stride_h + (long long)L * HD;
    __nv_bfloat16 *vc = (__nv_bfloat16 *)a.vcache + (long long)b * a.stride_b + (long long)kvh * a.stride_h + (long long)L * HD;
    constexpr int PER = HALF / 4;                  // four adjacent pairs per thread and pass
#pragma unroll 2
    for (int u = tid; u < wrows * PER; u += kShortThreads) {
      const int j = u / PER, i = (u % PER) * 4;
      uint2 k0 = make_uint2(0u, 0u), k1 = k0, v0 = k0, v1 = k0;    // rows behind the window: zero (a zero probability meets no NaN pattern)
      if (j < c) {
        const int r = bl * c + j;
        const float *src = a.qkv + (long long)r * a.ldq + qd + kvh * HD + i;
        const float4 x = __ldcg(reinterpret_cast<const float4 *>(src)), y = __ldcg(reinterpret_cast<const float4 *>(src + HALF));
        const float4 p = __ldcg(reinterpret_cast<const float4 *>(src + kvd)), q = __ldcg(reinterpret_cast<const float4 *>(src + kvd + HALF));
        const float4 *rp = reinterpret_cast<const float4 *>(a.rope + (long long)(L + j) * HALF + i);
        const float4 t0 = __ldg(rp), t1 = __ldg(rp + 1);
        const float s = rsqrtf(__ldcg(a.ss + r) / (float)a.dn + a.eps);
        const float x0 = x.x * s, x1 = x.y * s, x2 = x.z * s, x3 = x.w * s, y0 = y.x * s, y1 = y.y * s, y2 = y.z * s, y3 = y.w * s;
        k0 = make_uint2(pack2(x0 * t0.x - y0 * t0.y, x1 * t0.z - y1 * t0.w), pack2(x2 * t1.x - y2 * t1.y, x3 * t1.z - y3 * t1.w));
        k1 = make_uint2(pack2(x0 * t0.y + y0 * t0.x, x1 * t0.w + y1 * t0.z), pack2(x2 * t1.y + y2 * t1.x, x3 * t1.w + y3 * t1.z));
        v0 = make_uint2(pack2(p.x * s, p.y * s), pack2(p.z * s, p.w * s)); v1 = make_uint2(pack2(q.x * s, q.y * s), pack2(q.z * s, q.w * s));
        if (store) {
          *reinterpret_cast<uint2 *>(kc + (long long)j * HD + i) = k0; *reinterpret_cast<uint2 *>(kc + (long long)j * HD + i + HALF) = k1;
          *reinterpret_cast<uint2 *>(vc + (long long)j * HD + i) = v0; *reinterpret_cast<uint2 *>(vc + (long long)j * HD + i + HALF) = v1;
        }
      }
      const uint32_t o0 = piece(j, i >> 3, wsub) + (uint32_t)(i & 7) * 2u, o1 = piece(j, (i + HALF) >> 3, wsub) + (uint32_t)(i & 7) * 2u;
      *reinterpret_cast<uint2 *>(gen + (win_k - base) + o0) = k0; *reinterpret_cast<uint2 *>(gen + (win_k - base) + o1) = k1;
      *reinterpret_cast<uint2 *>(gen + (win_v - base) + o0) = v0; *reinterpret_cast<uint2 *>(gen + (win_v - base) + o1) = v1;
    }
  }
  __syncthreads();
  uint32_t qh[KS][4], ql[KS][4];
#pragma unroll
  for (int ks = 0; ks < KS; ++ks) {
    const uint4 h = reinterpret_cast<const uint4 *>(q_area)[ks * 32 + lane], w = reinterpret_cast<const uint4 *>(q_area)[(KS + ks) * 32 + lane];
    qh[ks][0] = h.x; qh[ks][1] = h.y; qh[ks][2] = h.z; qh[ks][3] = h.w;
    ql[ks][0] = w.x; ql[ks][1] = w.y; ql[ks][2] = w.z; ql[ks][3] = w.w;
  }

  const float sl2 = rsqrtf((float)HD) * 1.4426950408889634f;
  float m_run[2] = {-INFINITY, -INFINITY}, l_run[2] = {0.f, 0.f}, o[HD / 8][4];
#pragma unroll
  for (int n = 0; n < HD / 8; ++n)
#pragma unroll
    for (int i = 0; i < 4; ++i) o[n][i] = 0.f;
  bool ok = true;
  int issued = min(NS, n_mine);
  for (int i = 0; i < n_mine; ++i) {
    const int stage = i % NS, key0 = key0_of(i);
    if (!__all_sync(0xffffffffu, wait_bounded(smem_u32(&full_bar[warp][stage]), (uint32_t)(i / NS) & 1u))) { ok = false; break; }
    const uint32_t kb = ring + (uint32_t)stage * C::kTile, vb = kb + C::kHalf;
    const bool whole = key0 + kShortKeys <= L;
    if (!whole) {
      // values beyond the cached keys: whatever the slab holds there may be a NaN pattern
      unsigned char *vg = gen + (vb - base);
      for (int e = lane; e < (key0 + kShortKeys - L) * (HD / 8); e += 32)
        *reinterpret_cast<uint4 *>(vg + piece(L - key0 + e / (HD / 8), e % (HD / 8), C::kSub)) = make_uint4(0, 0, 0, 0);
      __syncwarp();
    }
    attend<HD, kShortKeys / 8>(kb, vb, C::kSub, qh, ql, o, m_run, l_run, sl2, lane, whole,
                               [&](int n, int x) { return key0 + n * 8 + t4 * 2 + (x & 1) < L; });
    __syncwarp();
    if (i + NS < n_mine) {
      if (lane == 0) { fence_proxy_async(); request(i + NS); }
      ++issued;
    }
  }
  if (has_win) {
    // 16-key blocks of the window, dealt to the warps behind the cached tiles
    const int j0 = min(q0 + g4, nq - 1) / group, j1 = min(q0 + g4 + 8, nq - 1) / group, j_last = min(q0 + 15, nq - 1) / group;
    for (int blk = (warp - n_cta % kShortWarps + kShortWarps) % kShortWarps; blk * 16 < wrows; blk += kShortWarps) {
      if (blk * 16 > j_last) break;
      attend<HD, 2>(win_k + (uint32_t)blk * 2048u, win_v + (uint32_t)blk * 2048u, wsub, qh, ql, o, m_run, l_run, sl2, lane, false,
                    [&](int n, int x) { return blk * 16 + n * 8 + t4 * 2 + (x & 1) <= (x >> 1 ? j1 : j0); });
    }
  }
#pragma unroll
  for (int hh = 0; hh < 2; ++hh) {
    l_run[hh] += __shfl_xor_sync(0xffffffffu, l_run[hh], 1);
    l_run[hh] += __shfl_xor_sync(0xffffffffu, l_run[hh], 2);
  }
  if (!__syncthreads_and(ok ? 1 : 0)) {
    // a tile did not arrive: no result; this warp's copies on their way are waited for (bounded)
    if (lane == 0) {
      atomicExch(a.err, 1u);
      const unsigned long long t0 = clock64();
      for (int i = 0; i < NS && i < issued; ++i)
        while (!mbar_try(smem_u32(&full_bar[warp][i]), last_copy_parity(issued, NS, i)))
          if ((unsigned long long)(clock64() - t0) > kSpinBudget / 4) break;
    }
    __syncthreads();
  }

  // ---- partial results of the warps
  {
    float *ob = obuf + warp * 16 * OLD;
#pragma unroll
    for (int n = 0; n < HD / 8; ++n) {
      *reinterpret_cast<float2 *>(ob + g4 * OLD + n * 8 + t4 * 2) = make_float2(o[n][0], o[n][1]);
      *reinterpret_cast<float2 *>(ob + (g4 + 8) * OLD + n * 8 + t4 * 2) = make_float2(o[n][2], o[n][3]);
    }
    if (t4 == 0) { ml[warp][g4] = make_float2(m_run[0], l_run[0]); ml[warp][g4 + 8] = make_float2(m_run[1], l_run[1]); }
  }
  __syncthreads();
  auto store = [&](int row, int c4, float4 v) {
    const int q = q0 + row, j = q / group, h = kvh * group + q - j * group;
    const long long at = (long long)(bl * c + j) * qd + h * HD + c4 * 4;
    const uint2 hi = make_uint2(pack2(v.x, v.y), pack2(v.z, v.w));
    __nv_bfloat16 *p = (__nv_bfloat16 *)a.out_pan + at;
    *reinterpret_cast<uint2 *>(p) = hi;
    *reinterpret_cast<uint2 *>(p + (long long)a.pan_rows * qd) =
        make_uint2(pack2(v.x - low_half(hi.x), v.y - high_half(hi.x)), pack2(v.z - low_half(hi.y), v.w - high_half(hi.y)));
  };
  for (int u = tid; u < 16 * (HD / 4); u += kShortThreads) {
    const int row = u / (HD / 4), c4 = u - row * (HD / 4);
    float M = -INFINITY;
#pragma unroll
    for (int k = 0; k < kShortWarps; ++k) M = fmaxf(M, ml[k][row].x);
    float den = 0.f;
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int k = 0; k < kShortWarps; ++k) {
      const float2 v = ml[k][row];
      const float w = v.x == -INFINITY ? 0.f : ex2((v.x - M) * sl2);
      const float4 x = *reinterpret_cast<const float4 *>(obuf + (k * 16 + row) * OLD + c4 * 4);
      den = fmaf(v.y, w, den);
      acc.x = fmaf(w, x.x, acc.x); acc.y = fmaf(w, x.y, acc.y); acc.z = fmaf(w, x.z, acc.z); acc.w = fmaf(w, x.w, acc.w);
    }
    if (ns == 1) {
      if (q0 + row < nq) {
        const float inv = 1.0f / den;
        store(row, c4, make_float4(acc.x * inv, acc.y * inv, acc.z * inv, acc.w * inv));
      }
    } else {
      *reinterpret_cast<float4 *>(obuf + row * OLD + c4 * 4) = acc;                     // only this thread reads these
      if (c4 == 0) ml_cta[row] = make_float2(M, den);
    }
  }
  if (ns > 1) {
    // ---- merge of the key splits through the cluster's shared memory
    __syncwarp();
    cluster_sync_all();
    const uint32_t ml_addr = smem_u32(ml_cta);
    for (int u = split * kShortThreads + tid; u < 16 * (HD / 4); u += ns * kShortThreads) {
      const int row = u / (HD / 4), c4 = u - row * (HD / 4);
      if (q0 + row >= nq) continue;
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
    __syncwarp();
    // The other splits may still be reading this CTA's memory.  (Relaxed: what was read has arrived, it is in the stores; a release
    // would wait for these too.)
    asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  }
}

// ------------------------------------------------------------------------------------ host side
template <int HD>
static cudaError_t short_config(cudaLaunchConfig_t &cfg, cudaLaunchAttribute (&attr)[2], int ns, int ny, int nz, size_t smem, bool pdl, cudaStream_t st) {
  static RisingLimit limit;
  const cudaError_t set = limit.raise(current_device_slot(), smem, [](size_t n) {
    return cudaFuncSetAttribute(attn_short_kernel<HD>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)n);
  });
  if (set != cudaSuccess) return set;
  memset(&cfg, 0, sizeof cfg);
  cfg.gridDim = dim3(ns, ny, nz); cfg.blockDim = dim3(kShortThreads); cfg.dynamicSmemBytes = smem; cfg.stream = st;
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

// Clusters of ns CTAs that run at the same time (B200, one CTA per SM: 74 of two, 45 of three, 33 of four, 26 22 15 15; two: 148 93 71 56 45 37 33).
// With two per SM a sixteenth is left out, because CTAs of the kernel in front still hold slots when they are placed (36 of 37 clusters of seven ran
// in two rounds).
template <int HD>
static int short_clusters(int ns, bool deep, int c) {
  static int known[kMaxDevices][9][2][4] = {};
  int &n = known[current_device_slot()][ns][deep][(c - 1) / 16];
  if (n == 0) {
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute attr[2];
    int fit = 0;
    if (short_config<HD>(cfg, attr, ns, 1, 1, short_smem<HD>(c, ShortCfg<HD>::stages(deep)), false, nullptr) != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&fit, attn_short_kernel<HD>, &cfg) != cudaSuccess || fit < 1) {
      (void)cudaGetLastError();
      fit = 1;
    }
    n = !deep && fit > 15 ? fit * 15 / 16 : fit;
  }
  return n;
}

template <int HD>
static cudaError_t launch_short_t(const KvTensorMap &map, ShortAttnArgs a, int tiles, int nqt, int nb, int n_sms, cudaStream_t st) {
  int ns;
  bool deep;
  short_plan(tiles, (long long)nb * a.hkv * nqt, HD, kShortWarps, n_sms, [&](int s, bool d) { return (long long)short_clusters<HD>(s, d, a.c); }, ns, deep);
  a.stages = ShortCfg<HD>::stages(deep);
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr[2];
  cudaError_t e = short_config<HD>(cfg, attr, ns, a.hkv * nqt, nb, short_smem<HD>(a.c, a.stages), a.pdl != 0, st);
  return e == cudaSuccess ? cudaLaunchKernelEx(&cfg, attn_short_kernel<HD>, *reinterpret_cast<const CUtensorMap *>(&map), a) : e;
}

// map: boxes of attn_stream_tile_keys() keys.
cudaError_t launch_attn_short(const KvTensorMap &map, const ShortAttnArgs &a, int nb, int max_len, int hd, int n_sms, cudaStream_t st) {
  if (nb < 1 || nb > 65535 || a.c < 1 || a.c > 64 || !a.err || !a.out_pan || (hd != 64 && hd != 128)) return cudaErrorInvalidValue;
  const int nqt = ((a.hq / a.hkv) * a.c + 15) / 16;
  if ((long long)a.hkv * nqt > 65535) return cudaErrorInvalidValue;
  const int tiles = (max_len + kShortKeys - 1) / kShortKeys;
  // One CTA per SM with 128 KB of tiles in flight, or two with half of that each (short_plan).  Measured, a step, one -> two: 7B, 2 x 16 rows over
  // 803 keys (64 units, clusters of 2 -> 4) 3042 -> 3022 us, 1 x 32 over 8000 4150 -> 3995; 13B, 2 x 16 over 4000 (80 units, 1 -> 3) 7439 ->
  // 6962; but 1 x 16 over 8000 (32 units, 4 -> 8) 3280 -> 3873; 13B, 1 x 16 over 8000 (40 units, 3 -> 7) 6434 -> 7084; 7B, 4 x 16 over 2048
  // (128 units, 1 -> 2) 4665 -> 4723.  head_dim 64: 1.1B, 1 x 16 over 8000 (4 -> 8) 1195 -> 1158.
  // Splits that do not all fit against the next fewer that do, 8 layers of 1.1B, one sequence: 10 rows over 1000 keys (20 units, 7 -> 6) 394 -> 359 us,
  // 12 rows (24, 6 -> 5) 394 -> 361, 18 rows (36, 4 -> 3) 454 -> 417, over 3000 (8 -> 6) 478 -> 436; 6 layers of 24 query and 8 kv heads of 128 (201 MB),
  // 32 rows over 3000 keys (48, 3 -> 5 with two CTAs per SM) 560 -> 466.
  return hd == 128 ? launch_short_t<128>(map, a, tiles, nqt, nb, n_sms, st) : launch_short_t<64>(map, a, tiles, nqt, nb, n_sms, st);
}

// The streaming pair reads faster where there is much to read (two CTAs of 96 KB of tiles per SM) but takes a second launch per layer, about
// 4 us.  Measured, a step, short -> pair, by 16-query units x 64-key tiles.  head_dim 128: 7B, 2 x 16 rows over 1500 keys (1536) 3125 us ->
// 3233; 4 x 16 over 2048 (4224) 4665 -> 4802; 1 x 16 over 8000 (4032) 3280 -> 3391; 4 x 8 over 4000 (8064) 4186 -> 4233; 16 x 1 over 1024 (8704) 3933
// -> 3931, over 2048 (16896) 5061 -> 4979.  More units than SMs leave the short kernel a second round: 5 x 8 over 3000 (160 units, 7680) 5488 -> 5306,
// over 2000 (5120) 4962 -> 4949 behind the chained launch.  head_dim 64: 1.1B, 16 x 4 over 1024 (2176) 1659 -> 1703; 1 x 16 over 8000 (4032) 1158 -> 1579;
// 4 x 16 over 4000 (8064) 2000 -> 1967; 16 x 4 over 8000 (16128) 2482 -> 2243.
bool attn_short_pays(int max_len, int c, int hq, int hkv, int nb, int hd, int n_sms) {
  const long long units = (long long)nb * hkv * (((long long)(hq / hkv) * c + 15) / 16);
  return units * ((max_len + c + 63) / 64) < (hd == 128 ? (units > n_sms ? 6000 : 8600) : 4600);
}

}  // namespace fc
