// A whole forward of a small fp32 model in one kernel: one thread-block cluster of sixteen CTAs, a hardware cluster barrier
// between dependent steps.
//
// At this size (a layer's weights are a few hundred KB, a few rows) nothing but latency counts: as separate launches a step
// of the 2-layer, 128-wide shape is 15 kernels of 3 to 20 us each, whose work is a microsecond.  Five barriers per layer
// remain (QKV | attention | O | gate/up | down), each a few hundred nanoseconds.
//
// A projection output is one warp's dot product over the whole k range (lanes stride over k, 8 rows at a time, one addition
// into the residual): no atomics, deterministic.  The rows are staged in shared memory once per CTA and step, with the RMSNorm gain
// applied and the row's sum of squares taken on the way.  The QKV step computes both elements of a rotary pair in one warp
// and so finishes q, k and v itself; gate and up of one feature share a warp as well.  Attention: one (row, head) per group
// of warps that deal the keys in blocks of eight.
#include <cstring>

#include "fc_accept.cuh"
#include "fc_ptx.cuh"

namespace fc {

namespace {
constexpr int kSmCtas = 16, kSmThreads = 1024, kSmWarps = kSmThreads / 32;
constexpr int kSmRows = 32;                          // rows staged at a time
constexpr int kSmallK = 1536;                        // widest input of a projection: the staged rows fill 192 KB

// Sums of eight per-lane values over the warp: lane returns the total of value lane >> 2.
__device__ __forceinline__ float sum8(float (&v)[8], int lane) {
#pragma unroll
  for (int o = 16, n = 4; o >= 4; o >>= 1, n >>= 1) {
    const bool up = lane & o;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      if (i >= n) break;
      const float give = up ? v[i] : v[i + n], keep = up ? v[i + n] : v[i];
      v[i] = keep + __shfl_xor_sync(0xffffffffu, give, o);
    }
  }
  float t = v[0];
  t += __shfl_xor_sync(0xffffffffu, t, 2);
  t += __shfl_xor_sync(0xffffffffu, t, 1);
  return t;
}
__device__ __forceinline__ float dot4(float4 a, float4 b, float acc) {
  return fmaf(a.w, b.w, fmaf(a.z, b.z, fmaf(a.y, b.y, fmaf(a.x, b.x, acc))));
}
}  // namespace

template <int ND>
__global__ void __launch_bounds__(kSmThreads, 1) small_forward_kernel(const __grid_constant__ SmallArgs a) {
  extern __shared__ __align__(16) float xs[];        // [kSmRows][max K]; the attention step's partial results
  __shared__ float s_rms[kSmRows];
  __shared__ unsigned long long best[kSmRows];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int cta = (int)cluster_rank();
  const int gw = warp * kSmCtas + cta;               // units go round the CTAs first
  constexpr int kUnits = kSmWarps * kSmCtas;
  constexpr int hd = ND * 32, half = hd >> 1;
  const int R = a.R, d = a.d, qd = a.hq * hd, F = a.f, group = a.hq / a.hkv;

  auto seq_of = [&](int r, int &b, int &j) { const int i = r / a.c; b = a.seq_map ? a.seq_map[i] : a.b0 + i; j = r - i * a.c; };
  // rows r0 .. r0 + n - 1 of src (gain == null: as they are) to shared memory, 1/rms of each
  auto stage = [&](const float *src, int ld, int K, const float *gain, int r0, int n) {
    __syncthreads();
    for (int i = warp; i < n; i += kSmWarps) {
      const float *p = src ? src + (long long)(r0 + i) * ld : a.emb + (long long)a.tokens[r0 + i] * d;
      float sq = 0.f;
      for (int k = lane * 4; k < K; k += 128) {
        float4 v = __ldcg(reinterpret_cast<const float4 *>(p + k));
        if (gain) {
          sq = dot4(v, v, sq);
          const float4 g = __ldg(reinterpret_cast<const float4 *>(gain + k));
          v.x *= g.x; v.y *= g.y; v.z *= g.z; v.w *= g.w;
        }
        *reinterpret_cast<float4 *>(xs + i * K + k) = v;
      }
      if (gain) {
        sq = warp_sum_f(sq);
        if (lane == 0) s_rms[i] = rsqrtf(sq / (float)d + a.eps);
      }
    }
    __syncthreads();
  };
  // dot products of two weight rows (the same twice: one) with eight staged rows; lane >> 2 is the row of the result
  auto dots = [&](const float *w0, const float *w1, int K, const float *x0, float &s0, float &s1) {
    float p[8], q[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) p[i] = q[i] = 0.f;
    for (int k = lane * 4; k < K; k += 128) {
      const float4 u = __ldg(reinterpret_cast<const float4 *>(w0 + k));
      float4 v = u;
      if (w1) v = __ldg(reinterpret_cast<const float4 *>(w1 + k));
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const float4 x = *reinterpret_cast<const float4 *>(x0 + i * K + k);
        p[i] = dot4(u, x, p[i]);
        if (w1) q[i] = dot4(v, x, q[i]);
      }
    }
    s0 = sum8(p, lane);
    s1 = w1 ? sum8(q, lane) : 0.f;
  };

  // This warp's first weight row of a coming step on its way into the first-level cache while the barrier in front of
  // that step is waited for: nobody waits for these loads.
  auto touch = [&](const float *row, int K) {
    for (int k = lane * 4; k < K; k += 128) {
      float t;
      asm volatile("ld.global.nc.f32 %0, [%1];" : "=f"(t) : "l"(row + k));
    }
  };
  // the first row of the rotary pair that is unit u of the QKV step
  auto pair_row = [&](const SmallLayer &w, int u) -> const float * {
    const int h = u / half, i = u - h * half;
    return (h < a.hq ? w.wq + (long long)h * hd * d : h < a.hq + a.hkv ? w.wk + (long long)(h - a.hq) * hd * d : w.wv + (long long)(h - a.hq - a.hkv) * hd * d) + (long long)i * d;
  };
  const int n_pairs = (a.hq + 2 * a.hkv) * half;

  for (int l = 0; l < a.n_layers; ++l) {
    const SmallLayer &w = a.layers[l];
    const float *x_in = l == 0 ? nullptr : a.x;                   // layer 0 reads the embedding rows themselves
    float *kc = a.kv + (long long)(2 * l) * a.half_stride, *vc = kc + a.half_stride;
    // ---- q, k, v: a unit is a rotary pair of one head
    for (int r0 = 0; r0 < R; r0 += kSmRows) {
      const int n = min(kSmRows, R - r0);
      stage(x_in, d, d, w.g_attn, r0, n);
      for (int u = gw; u < n_pairs; u += kUnits) {
        const int h = u / half, i = u - h * half;
        const float *m = pair_row(w, u);
        for (int c0 = 0; c0 < n; c0 += 8) {
          const int rr = c0 + (lane >> 2), r = r0 + min(rr, n - 1);
          int b, j;
          seq_of(r, b, j);
          const int pos = a.kv_len[b] + j;                          // on its way, with the rotation, beside the weights
          const float2 rot = __ldg(a.rope + (long long)pos * half + i);
          float v0, v1;
          dots(m, m + (long long)half * d, d, xs + c0 * d, v0, v1);
          if ((lane & 3) || rr >= n) continue;
          v0 *= s_rms[rr]; v1 *= s_rms[rr];
          if (h < a.hq + a.hkv) {
            const float o0 = v0 * rot.x - v1 * rot.y, o1 = v0 * rot.y + v1 * rot.x;
            v0 = o0; v1 = o1;
          }
          float *dst = h < a.hq ? a.q + (long long)r * qd + h * hd
                                : (h < a.hq + a.hkv ? kc + (long long)(h - a.hq) * a.stride_h : vc + (long long)(h - a.hq - a.hkv) * a.stride_h) + (long long)b * a.stride_b + (long long)pos * hd;
          dst[i] = v0; dst[i + half] = v1;
        }
      }
    }
    if (!a.with_head && l + 1 == a.n_layers) break;                 // rows that are only cached: nothing reads what follows
    if (gw < d) touch(w.wo + (long long)gw * qd, qd);
    cluster_sync_all();
    // ---- attention: a (row, head) per group of warps, keys dealt in blocks of eight
    {
      const int per_cta = (R * a.hq + kSmCtas - 1) / kSmCtas;
      int wpu = kSmWarps;                                           // warps per unit
      while (wpu > 1 && kSmWarps / wpu < per_cta) wpu >>= 1;
      const int upc = kSmWarps / wpu, sub = warp % wpu;                          // units at a time per CTA
      const float scale = rsqrtf((float)hd);
      float *part = xs;                                             // [warp][hd + 2]
      for (int u0 = 0; u0 < per_cta; u0 += upc) {
        const int u = (u0 + warp / wpu) * kSmCtas + cta;
        const bool live = u < R * a.hq;
        float m = -INFINITY, lsum = 0.f, o[ND] = {};
        const int r = live ? u / a.hq : 0, h = live ? u - r * a.hq : 0;
        if (live) {
          int b, j;
          seq_of(r, b, j);
          const int n_keys = a.kv_len[b] + j + 1;
          const float *kp = kc + (long long)b * a.stride_b + (long long)(h / group) * a.stride_h + lane;
          const float *vp = vc + (long long)b * a.stride_b + (long long)(h / group) * a.stride_h + lane;
          float q[ND];
#pragma unroll
          for (int e = 0; e < ND; ++e) q[e] = __ldcg(a.q + (long long)r * qd + h * hd + e * 32 + lane) * scale;
          for (int k0 = sub * 8; k0 < n_keys; k0 += wpu * 8) {
            float s[8], v[8][ND];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
              s[i] = 0.f;
#pragma unroll
              for (int e = 0; e < ND; ++e) v[i][e] = 0.f;
              if (k0 + i < n_keys) {
#pragma unroll
                for (int e = 0; e < ND; ++e) {
                  s[i] = fmaf(q[e], __ldcg(kp + (long long)(k0 + i) * hd + e * 32), s[i]);
                  v[i][e] = __ldcg(vp + (long long)(k0 + i) * hd + e * 32);
                }
              }
            }
            const float mine = sum8(s, lane);                       // score of key k0 + (lane >> 2)
            const float sc = k0 + (lane >> 2) < n_keys ? mine : -INFINITY;
            float mx = fmaxf(m, sc);
#pragma unroll
            for (int e = 4; e < 32; e <<= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, e));
            const float corr = m == -INFINITY ? 0.f : expf(m - mx), p = sc == -INFINITY ? 0.f : expf(sc - mx);
            float ps = p;
#pragma unroll
            for (int e = 4; e < 32; e <<= 1) ps += __shfl_xor_sync(0xffffffffu, ps, e);
            lsum = lsum * corr + ps;
            m = mx;
#pragma unroll
            for (int e = 0; e < ND; ++e) o[e] *= corr;
#pragma unroll
            for (int i = 0; i < 8; ++i) {
              const float pi = __shfl_sync(0xffffffffu, p, i * 4);
#pragma unroll
              for (int e = 0; e < ND; ++e) o[e] = fmaf(pi, v[i][e], o[e]);
            }
          }
        }
        __syncthreads();                                            // the buffer's last readers are done
        float *mine = part + warp * (hd + 2);
#pragma unroll
        for (int e = 0; e < ND; ++e) mine[e * 32 + lane] = o[e];
        if (lane == 0) { mine[hd] = m; mine[hd + 1] = lsum; }
        __syncthreads();
        if (live && sub == 0) {
          float M = -INFINITY, den = 0.f, acc[ND] = {};
          for (int i = 0; i < wpu; ++i) M = fmaxf(M, mine[i * (hd + 2) + hd]);
          for (int i = 0; i < wpu; ++i) {
            const float *pi = mine + i * (hd + 2);
            if (pi[hd + 1] == 0.f) continue;
            const float wgt = expf(pi[hd] - M);
            den = fmaf(pi[hd + 1], wgt, den);
#pragma unroll
            for (int e = 0; e < ND; ++e)
              acc[e] = fmaf(wgt, pi[e * 32 + lane], acc[e]);
          }
          const float inv = 1.0f / den;
#pragma unroll
          for (int e = 0; e < ND; ++e)
            a.attn[(long long)r * qd + h * hd + e * 32 + lane] = acc[e] * inv;
        }
      }
    }
    cluster_sync_all();
    // ---- x += attn . Wo
    auto add_to_x = [&](const float *src, int K, const float *m, bool from_emb, auto &&next) {
      for (int r0 = 0; r0 < R; r0 += kSmRows) {
        const int n = min(kSmRows, R - r0);
        stage(src, K, K, nullptr, r0, n);
        for (int u = gw; u < d; u += kUnits)
          for (int c0 = 0; c0 < n; c0 += 8) {
            const int rr = c0 + (lane >> 2), r = r0 + min(rr, n - 1);
            float *x = a.x + (long long)r * d + u;
            const float before = from_emb ? a.emb[(long long)a.tokens[r] * d + u] : __ldcg(x);
            float v, none;
            dots(m + (long long)u * K, nullptr, K, xs + c0 * K, v, none);
            if ((lane & 3) || rr >= n) continue;
            *x = before + v;
          }
      }
      next();
      cluster_sync_all();
    };
    add_to_x(a.attn, qd, w.wo, l == 0, [&] {
      if (gw < F) { touch(w.w_gate + (long long)gw * d, d); touch(w.w_up + (long long)gw * d, d); }
    });
    // ---- silu(gate) * up
    for (int r0 = 0; r0 < R; r0 += kSmRows) {
      const int n = min(kSmRows, R - r0);
      stage(a.x, d, d, w.g_ffn, r0, n);
      for (int u = gw; u < F; u += kUnits)
        for (int c0 = 0; c0 < n; c0 += 8) {
          float g, up;
          dots(w.w_gate + (long long)u * d, w.w_up + (long long)u * d, d, xs + c0 * d, g, up);
          const int rr = c0 + (lane >> 2);
          if ((lane & 3) || rr >= n) continue;
          g *= s_rms[rr]; up *= s_rms[rr];
          a.h[(long long)(r0 + rr) * F + u] = (g / (1.0f + expf(-g))) * up;
        }
    }
    if (gw < d) touch(w.w_down + (long long)gw * F, F);
    cluster_sync_all();
    add_to_x(a.h, F, w.w_down, false, [&] {
      if (l + 1 < a.n_layers) {
        if (gw < n_pairs) { const float *m = pair_row(a.layers[l + 1], gw); touch(m, d); touch(m + (long long)half * d, d); }
      } else if (a.with_head && gw < a.vocab) {
        touch(a.lm_head + (long long)gw * d, d);
      }
    });
  }
  if (!a.with_head) return;
  // ---- LM head, greedy token per row
  for (int r0 = 0; r0 < R; r0 += kSmRows) {
    const int n = min(kSmRows, R - r0);
    stage(a.x, d, d, a.g_final, r0, n);
    if (tid < kSmRows) best[tid] = 0ull;
    __syncthreads();
    for (int u = gw; u < a.vocab; u += kUnits)
      for (int c0 = 0; c0 < n; c0 += 8) {
        const int rr = c0 + (lane >> 2), r = r0 + min(rr, n - 1);
        const int favoured = a.perm ? a.perm[a.tokens[r]] : -1;
        float v, none;
        dots(a.lm_head + (long long)u * d, nullptr, d, xs + c0 * d, v, none);
        if ((lane & 3) || rr >= n) continue;
        float logit = v * s_rms[rr];
        if (favoured == u) logit += a.beta;
        if (a.logits) a.logits[(long long)r * a.vocab + u] = logit;
        atomicMax(&best[rr], ((unsigned long long)ordered_key_u(logit) << 32) | (unsigned long long)(0xFFFFFFFFu - (unsigned int)u));
      }
    __syncthreads();
    if (tid < n) atomicMax(&a.accept.amax_clear[r0 + tid], best[tid]);
  }
  cluster_sync_all();
  // ---- verification, commit, shift, refill: one warp per sequence
  for (int i = gw; i < a.accept.nb; i += kUnits) accept_warp(a.accept, i, lane);
}

// Models whose steps this kernel is made for: sixteen SMs hold and stream their layers.  Measured, this kernel against the
// separate ones, per step: 2 layers, d 128, ffn 512 (1 MB of weights a layer), 8 rows over 64 keys 41 against 211 us, 4 x 16
// rows over 200 keys 150 against 1200; 8 layers, d 256, ffn 768 (3.3 MB), 8 rows over 512 keys 271 against 1144, 4 x 16 rows
// 1530 against 7142; a prompt of 512 8.1 against 56.7 ms; 4 layers, d 512, ffn 1024 (10 MB), 1 row 189 against 337, 8 rows 218
// against 803.  At 34 MB a layer and 131 MB of LM head one row costs more here (851 against 810).
bool small_model_fits(int d, int qd, int kvd, int f, int hd, int vocab, int n_layers) {
  const long long layer = (long long)d * (2 * qd + 2 * kvd + 3 * f) * 4;
  return n_layers <= kSmallLayers && d <= kSmallK && qd <= kSmallK && f <= kSmallK && layer <= (16 << 20) &&
         (long long)vocab * d * 4 <= (16 << 20) && hd <= 128;
}

// Whether a forward of R rows over `keys` keys takes this kernel.  Every (row, head) reads its keys for itself here, on sixteen SMs,
// where the attention of the separate kernels shares a tile of keys among all queries of a kv head and uses every SM; what
// those lose is 9 to 21 us per row and layer in their projections.  Measured, one kernel / separate ones: 2 layers of 4 heads x 32, 1024
// rows, 512 keys 2.6 / 17.8 ms, 2048 keys 7.0 / 18.1, 8192 keys 27.1 / 19.0; 8 layers of 8 x 64, 256 rows, 2048 keys 20.0 / 31.3, 8192
// keys 69.6 / 37.6; 4 layers of 4 x 128, 256 rows, 2048 keys 10.0 / 22.1, 8192 keys 27.5 / 24.7.  The lines cross at 22, 28 and
// 27 thousand keys x heads; with up to 32 rows, where the separate kernels fill few SMs, at 50 to 107 thousand (8 x 64, 8192 keys: 1
// row 0.64 / 0.97 ms, 32 rows 7.6 / 9.4).
bool small_forward_pays(int R, int heads, int keys) { return (long long)heads * keys <= (R < 64 ? 66000 : 24000); }

static size_t small_smem(int d, int qd, int f, int hd) {
  const int k = d > qd ? (d > f ? d : f) : (qd > f ? qd : f);
  const size_t rows = (size_t)kSmRows * k * 4, att = (size_t)kSmWarps * (hd + 2) * 4;
  return rows > att ? rows : att;
}

// Launch configuration; the opt-ins are the same for every model, so that contexts do not undo each other's.
template <int ND>
static cudaError_t small_config(cudaLaunchConfig_t &cfg, cudaLaunchAttribute &attr, size_t smem, cudaStream_t st) {
  static bool attr_done[kMaxDevices] = {false};
  const int dev = current_device_slot();
  if (!attr_done[dev]) {
    cudaError_t e = cudaFuncSetAttribute(small_forward_kernel<ND>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmRows * kSmallK * 4);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(small_forward_kernel<ND>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    attr_done[dev] = true;
  }
  memset(&cfg, 0, sizeof cfg);
  cfg.gridDim = dim3(kSmCtas); cfg.blockDim = dim3(kSmThreads); cfg.dynamicSmemBytes = smem; cfg.stream = st;
  attr.id = cudaLaunchAttributeClusterDimension;
  attr.val.clusterDim.x = kSmCtas; attr.val.clusterDim.y = 1; attr.val.clusterDim.z = 1;
  cfg.attrs = &attr; cfg.numAttrs = 1;
  return cudaSuccess;
}

template <int ND>
static cudaError_t launch_small_t(const SmallArgs &a, size_t smem, cudaStream_t st) {
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr;
  cudaError_t e = small_config<ND>(cfg, attr, smem, st);
  return e == cudaSuccess ? cudaLaunchKernelEx(&cfg, small_forward_kernel<ND>, a) : e;
}

cudaError_t launch_small_forward(const SmallArgs &a, cudaStream_t st) {
  const size_t smem = small_smem(a.d, a.hq * a.hd, a.f, a.hd);
  if (a.hd == 32) return launch_small_t<1>(a, smem, st);
  if (a.hd == 64) return launch_small_t<2>(a, smem, st);
  if (a.hd == 128) return launch_small_t<4>(a, smem, st);
  return cudaErrorInvalidValue;
}

template <int ND>
static int small_clusters_t(size_t smem) {
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr;
  int n = 0;
  if (small_config<ND>(cfg, attr, smem, nullptr) != cudaSuccess || cudaOccupancyMaxActiveClusters(&n, small_forward_kernel<ND>, &cfg) != cudaSuccess) {
    (void)cudaGetLastError();
    return 0;
  }
  return n;
}

// A cluster of sixteen is beyond the portable eight: not every device (or part of one) has sixteen SMs in one group.
bool small_cluster_fits(int d, int qd, int f, int hd) {
  const size_t smem = small_smem(d, qd, f, hd);
  return (hd == 32 ? small_clusters_t<1>(smem) : hd == 64 ? small_clusters_t<2>(smem) : hd == 128 ? small_clusters_t<4>(smem) : 0) > 0;
}

}  // namespace fc
