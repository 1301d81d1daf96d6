// Internal declarations shared by the CUDA sources of the Jacobi-window decode library.
#pragma once
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "fastcot.h"

namespace fc {

// ---- activation transform applied while an fp32 buffer is staged as the GEMM's row operand ----
enum ProOp : int {
  PRO_NONE = 0,      // x
  PRO_GAIN = 1,      // x * gain[k]                (RMSNorm gain; the 1/rms row factor is applied by the consumer)
  PRO_SILU_MUL = 2   // silu(s_r * g) * (s_r * u)  (SwiGLU on gate/up accumulators that still lack 1/rms)
};
enum EpiOp : int {
  EPI_ATOMIC_ADD = 0,  // y[r, n] += acc  (split-K partial sums, or += onto the residual stream)
  EPI_ARGMAX = 1       // logits = s_r * acc + bias; per-row running (max, lowest index) via 64-bit atomicMax
};

constexpr int kMaxMats = 3;

struct GemmArgs {
  // row operand: fp32 [R, K] with leading dimension ldx
  const float *x;
  const float *x2;        // PRO_SILU_MUL: the "up" half (x is the "gate" half)
  int ldx;
  const void *gain;       // PRO_GAIN: [K] in the weight dtype
  const float *ss_in;     // PRO_SILU_MUL: per-row sum of squares of the normalised input; s_r = rsqrt(ss/dn + eps)
  float *ss_out;          // PRO_GAIN: if non-null, sum_k x[r,k]^2 is accumulated here (once per k)
  float eps;
  int dn;                 // width the sums of squares are means over (d_model)
  // weights: up to three matrices [n_rows[m], K], outputs concatenated at column offsets y_off[m]
  const void *w[kMaxMats];
  int ldw;                // row pitch of the weight matrices in elements (0: K) - a column slice of a wider matrix
  int n_rows[kMaxMats];
  int y_off[kMaxMats];
  int n_mats;
  float *y;
  int ldy;
  int R, K;
  // EPI_ARGMAX
  const int32_t *tokens;          // [R] input token of each row (bias lookup)
  const int32_t *perm;            // [vocab] or null
  float beta;
  unsigned long long *amax;       // [R] packed (ordered logit << 32 | ~index)
  float *logits;                  // optional dump [R, vocab]
  int vocab;
  // more than 16 rows: bf16 panel [2][pan_rows][K] (high parts, then low parts) that the launch fills with pro(x) once
  // and streams by TMA; with the argmax epilogue ss_out then holds the row sums of squares the epilogue reads
  void *pan;
  int pan_rows;
  int pan_ready;                  // the panel already holds pro(x), written by the kernel before this launch: no conversion
};

struct ZeroList {       // buffers a kernel clears on the side (fp32 words)
  float *p[4];
  unsigned long long n[4];
};

struct RopeArgs {
  float *qkv;             // [R, ldq] accumulators: q | k | v, unscaled by 1/rms; cleared after reading
  int ldq;
  const float *ss;        // [R] sums of squares for the 1/rms factor
  float eps; int dn;
  const int32_t *kv_len;  // [batch] device
  const int32_t *seq_map; // optional [nb] device: the sequence behind row block i (null: b0 + i)
  int b0, nb, c;          // rows r = i * c + j for row block i
  int hq, hkv, hd;
  const float2 *rope;     // [max_seq][hd/2] (cos, sin) of position * theta^(-2i/hd), built on the host
  void *q_out;            // [R, hq*hd] in the cache dtype
  void *kcache, *vcache;  // layer base; element strides below
  long long stride_b, stride_h;   // per sequence, per kv head (elements); token stride is hd
  ZeroList z;
};

struct AttnArgs {
  const void *q;          // [R, hq*hd] cache dtype, already rotated
  const void *kcache, *vcache;
  long long stride_b, stride_h;
  const int32_t *kv_len;
  const int32_t *seq_map; // optional [nb] device: the sequence behind row block i (null: b0 + i)
  int b0, nb, c, hq, hkv;
  int nsplit;
  float *part_o;          // [R*hq, nsplit, hd]
  float *part_ml;         // [R*hq, nsplit, 2]
  unsigned int *counters; // [batch*hkv], zero on entry, zero on exit
  float *out;             // [R, hq*hd] fp32
  ZeroList z;
};

struct KvTensorMap { alignas(64) unsigned char opaque[128]; };   // storage of one TMA tensor map (CUtensorMap)

struct FusedAttnArgs {   // bf16: rotary embedding + K/V write + window attention in one kernel
  const float *qkv;       // [R, ldq] fp32 accumulators (q | k | v) lacking 1/rms; read only
  int ldq;
  const float *ss;        // [R] sums of squares for 1/rms; read only
  float eps; int dn;
  const float2 *rope;     // [max_seq][hd/2] (cos, sin) of position * theta^(-2i/hd)
  unsigned int c_magic;   // ceil(2^32 / c): q / c == umulhi(q, c_magic) for the small q used here
  void *kcache, *vcache;  // layer base (the window's own rows are stored through these)
  long long stride_b, stride_h;   // per sequence, per kv head (elements); stride_b == hkv * stride_h
  int k_plane0, v_plane0; // plane (= [max_seq][hd] matrix of one sequence and kv head) of sequence 0, kv head 0 in the
                          // K and the V tensor map: cached tiles are fetched by TMA from plane0 + b * hkv + kvh
  const int32_t *kv_len;
  const int32_t *seq_map; // optional [nb] device: the sequence behind row block i (null: b0 + i)
  int b0, nb, c, hq, hkv;
  int nsplit;             // CTAs (one thread-block cluster, <= 8) per (sequence, kv head, query-tile group)
  int qt;                 // 16-row query tiles per CTA: 1, 2 or 4
  int stages;             // K/V ring stages (set by the launcher)
  int pdl;                // launched as a programmatic dependent of the previous kernel
  unsigned int *err;      // device error word, raised when a bounded wait gives up
  float *out;             // [R, hq*hd] fp32
  // instead of `out`: the result as the bf16 pair high + low in the activation panel [2][pan_rows][hq*hd] that the output
  // projection streams by TMA (more than 16 rows per forward), which then needs no conversion pass of its own
  void *out_pan;
  int pan_rows;
  ZeroList z;
};

// The rows of a forward as runs of consecutive positions of one sequence each.  n == 0: every sequence has c rows, row
// block i belongs to sequence seq_map[i] (null: b0 + i).  n > 0: segment i is rows row0[i] .. row0[i + 1) of sequence
// seq[i].  Position of a row: kv_len[sequence] + its index in the run.
constexpr int kMaxSegs = 64;
struct RowSegs {
  int n, b0, c;
  const int32_t *seq_map;
  int seq[kMaxSegs], row0[kMaxSegs + 1];
};

struct QkvFinishArgs {    // bf16: QKV accumulators -> rotated queries (high + low) and K/V rows in the cache
  const float *qkv;       // [R, ldq] fp32 accumulators (q | k | v) lacking 1/rms; read only
  int ldq;
  const float *ss;        // [R] sums of squares for 1/rms
  float eps; int dn;
  const float2 *rope;     // [max_seq][hd/2] (cos, sin)
  const int32_t *kv_len;
  RowSegs segs;
  int hq, hkv, hd;
  void *q;                // bf16 high + low in MMA operand order, q_tiles tiles of 16 queries per kv head
  int q_tiles;
  void *kcache, *vcache;  // layer base
  long long stride_b, stride_h;
  int pdl;
  ZeroList z;
};

struct StreamAttnArgs {   // bf16: window attention over rows whose K/V are in the cache
  const void *q;          // as written by qkv_finish_kernel
  int q_tiles;
  const int32_t *kv_len;
  RowSegs segs;
  int hq, hkv;
  int k_plane0, v_plane0; // as in FusedAttnArgs
  unsigned int *err;
  float *out;             // [R, hq * hd] fp32, or
  void *out_pan;          // the bf16 pair [2][pan_rows][hq * hd]
  int pan_rows;
  int spare;              // behind a persistent launch: key splits leave room beside that kernel's last CTAs
  int pdl;
};

struct ShortAttnArgs {    // bf16: as FusedAttnArgs, for few queries over short caches (k_attn_short.cu); the result is the bf16 pair out_pan
  const float *qkv; int ldq;
  const float *ss; float eps; int dn;
  const float2 *rope;
  void *kcache, *vcache; long long stride_b, stride_h;
  int k_plane0, v_plane0;
  const int32_t *kv_len, *seq_map;
  int b0, c, hq, hkv;
  unsigned int *err;
  void *out_pan; int pan_rows;
  int stages;             // tiles in flight per warp (set by the launcher)
  int pdl;
};

struct AcceptArgs {
  int32_t *window;                 // [batch, c] in/out
  const unsigned long long *amax;  // packed argmax per row, or null
  unsigned long long *amax_clear;  // cleared after reading (may be null)
  const int32_t *argmax;           // plain argmax per row (used when amax is null)
  int32_t *kv_len, *n_gen, *done;  // [batch]; done may be null
  int32_t *accepted_count, *accepted_tokens;   // [batch], [batch, c]
  const int32_t *prompt, *prompt_lens;
  int32_t *out_tokens;             // [batch, out_stride] or null
  int out_stride;
  int b0, nb, c, p_stride, refill, pad_id;
  const int32_t *seq_map;          // optional [nb] device: the sequence behind row block i (null: b0 + i); rows of the
                                   // forward (amax / argmax) are indexed by row block, sequence state by sequence
  int max_tokens, eos_id;          // max_tokens <= 0: unlimited
  int commit;                      // 0: leave kv_len / n_gen / window untouched (latency measurement)
  unsigned int *err_inject;        // test aid: when non-null the kernel raises this error word (no wait involved)
  // what the host wants to know, written to its (pinned) memory as well; all null: nothing
  int32_t *host_count, *host_tokens, *host_window, *host_err;
  const unsigned int *err;         // the device error word behind host_err
};

// A small fp32 model's forward as one kernel (k_small.cu).
constexpr int kSmallLayers = 16;
struct SmallLayer { const float *wq, *wk, *wv, *wo, *w_gate, *w_up, *w_down, *g_attn, *g_ffn; };
struct SmallArgs {
  SmallLayer layers[kSmallLayers];
  int n_layers, d, hq, hkv, hd, f, vocab;
  const float *emb, *g_final, *lm_head;
  float eps;
  const float2 *rope;
  const int32_t *tokens;           // [R]
  const int32_t *kv_len, *seq_map; // row block i belongs to sequence seq_map[i] (null: b0 + i)
  int b0, c, R;
  float *kv;                       // K and V planes of a layer half_stride elements apart
  long long half_stride, stride_b, stride_h;
  float *x, *q, *attn, *h;         // [R, d], [R, qd], [R, qd], [R, f]
  int with_head;
  const int32_t *perm; float beta; float *logits;
  AcceptArgs accept;               // with_head: runs behind the LM head; accept.amax_clear is the argmax buffer, zero on entry
};
bool small_model_fits(int d, int qd, int kvd, int f, int hd, int vocab, int n_layers);
bool small_cluster_fits(int d, int qd, int f, int hd);      // the device can hold the kernel's cluster
bool small_forward_pays(int R, int heads, int keys);
cudaError_t launch_small_forward(const SmallArgs &a, cudaStream_t st);

struct EmbedArgs {
  const int32_t *tokens;   // [R], or with segs.n > 0 [sequence][t_stride]: row j of a segment is token kv_len[sequence] + j
  RowSegs segs;
  const int32_t *kv_len;
  int t_stride;
  const void *emb;         // [vocab, d]
  float *x;                // [R, d]
  int R, d;
  ZeroList z;
};

// Function attributes (dynamic shared memory opt-in, cluster size) are per device: launchers remember what they
// have set per device ordinal.
constexpr int kMaxDevices = 64;
inline int current_device_slot() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0) dev = 0;
  return dev % kMaxDevices;
}

// ---- launchers (each returns the cudaError_t of the launch) ----
cudaError_t launch_embed(const EmbedArgs &a, int dtype, cudaStream_t st);
cudaError_t launch_gemm_simt(const GemmArgs &a, int dtype, int pro, int epi, cudaStream_t st);
cudaError_t launch_rope_kv(const RopeArgs &a, int dtype, cudaStream_t st);
cudaError_t launch_attn(const AttnArgs &a, int dtype, int hd, cudaStream_t st);
cudaError_t launch_attn_fused(const KvTensorMap &kmap, const KvTensorMap &vmap, const FusedAttnArgs &a, int hd, cudaStream_t st);
// 3-d tensor map (head_dim, max_seq, planes) over bf16 K or V planes laid out [plane][max_seq][head_dim] from `base`.
// box_keys: keys per box.
cudaError_t make_kv_tensor_map(KvTensorMap *out, const void *base, int hd, int max_seq, long long planes, int box_keys);
cudaError_t launch_qkv_finish(const QkvFinishArgs &a, int R, cudaStream_t st);
// map: boxes of attn_stream_tile_keys() keys; max_rows / max_len: the longest segment and (a bound on) the longest cache
cudaError_t launch_attn_stream(const KvTensorMap &map, const StreamAttnArgs &a, int nseg, int max_rows, int max_len, int hd,
                               int n_sms, cudaStream_t st);
cudaError_t launch_attn_short(const KvTensorMap &map, const ShortAttnArgs &a, int nb, int max_len, int hd, int n_sms, cudaStream_t st);
bool attn_short_pays(int max_len, int c, int hq, int hkv, int nb, int hd, int n_sms);      // against the streaming pair, behind the one-writer projections
bool attn_stream_pays(int max_len, int c, int hq, int hkv, int nb);
int attn_stream_tile_keys();
size_t attn_stream_q_tiles(int rows, int group, int nseg);      // tiles per kv head for `rows` rows in nseg segments
int attn_fused_tile_keys();
// Grid of the fused attention kernel: splits per (sequence, kv head, query-tile group) and query tiles per CTA.
void fused_attn_plan(int max_len, int c, int hq, int hkv, int nb, int hd, int n_sms, int &nsplit, int &qt);
int attn_fused_max_rows();   // most window rows per sequence the fused kernel takes in one launch
cudaError_t launch_accept(const AcceptArgs &a, cudaStream_t st);
// dst[i * c + j] = window[seq_map[i] * c + j]: the token rows of a forward over the sequences seq_map[0 .. nb-1]
cudaError_t launch_gather_rows(int32_t *dst, const int32_t *window, const int32_t *seq_map, int nb, int c, cudaStream_t st);
int attn_tile_keys(int dtype, int hd);   // keys per split tile

// Standalone window attention on caller-supplied scratch (shared by the op-level entry points).
size_t window_attention_scratch_bytes(int batch, int c, int hq, int hkv, int hd, int max_len, int dtype);
int run_window_attention(const void *q, const void *kcache, const void *vcache, const int32_t *kv_len, float *out,
                         int batch, int c, int hq, int hkv, int hd, int max_seq, int max_len, int dtype,
                         void *scratch, size_t scratch_bytes, cudaStream_t st);

// tcgen05 path (bf16 only).  `maps` points at prebuilt tensor maps for the weight matrices.
struct UmmaPlan;
UmmaPlan *umma_plan_create(const GemmArgs &a, int pro, int epi, int n_sms, unsigned int *err_word,
                           char *err, int errlen);
void umma_plan_destroy(UmmaPlan *p);
// x/x2/y/ss pointers and R may differ per launch from those the plan was created with.
// claim: one zeroed word per projection of the launch (the work-claim counters).
// zero (optional): buffers the launch clears at its start, once the previous kernel is complete; only for buffers that
// nothing reads before a later kernel or a phase behind a grid barrier of this launch accumulates into them.
// cta_pairs: with 128-row blocks in panel mode and weight matrices of whole 256-row tiles, run as clusters of two
// CTAs that share a tile (tcgen05 cta_group::2).
cudaError_t launch_gemm_umma(const UmmaPlan *p, const GemmArgs &a, unsigned int *claim, unsigned int *bar_b,
                             const ZeroList *zero, int pdl, cudaStream_t st, int cta_pairs = 0);
// What other launchers need of a plan: tensor maps (boxes of 64 k x 128 rows), rows and output offsets of the matrices.
void umma_plan_view(const UmmaPlan *p, CUtensorMap *maps, const void **w, int *n_rows, int *y_off, int &n_mats, int &K, unsigned int *&err);
// Tensor map over 2 * pan_rows rows of K elements (bf16; an activation pair, or a weight matrix), boxes of 64 k x box_rows.
cudaError_t make_pair_tensor_map(CUtensorMap *out, const void *pan, int pan_rows, int K, int box_rows);

// ---- many rows: one dense GEMM per projection (k_bulk.cu); every weight matrix a whole number of 256-row tiles
enum BulkEpi : int {
  BULK_STORE = 0,     // y = acc
  BULK_ADD = 1,       // y += acc (the residual)
  BULK_SWIGLU = 2,    // plan of gate and up: silu(s g) * (s u) as the pair out_pan, s = 1/rms from ss
  BULK_HEAD = 3       // logits = s * acc + bias; per-row (max, lowest index)
};
struct BulkArgs {
  const void *pan;        // activation pair [2][pan_rows][K]
  int pan_rows, R;
  float *y; int ldy;
  const float *ss; float eps; int dn;
  void *out_pan;          // [2][pan_rows][d_ffn]
  void *slots;            // bulk_slot_bytes(): pieces of tiles that several pairs work on
  unsigned int *arrived;  // kBulkArrived words, zero before the first launch; every launch leaves them zero
  const int32_t *tokens, *perm; float beta; unsigned long long *amax; float *logits;
  int split;              // add up as the chained launch does (k_bulk.cu)
};
constexpr int kBulkPairs = 80;                       // CTA pairs the slots are laid out for
constexpr int kBulkArrived = kBulkPairs * 16;        // fewer units than pairs are ever shared; two ranks, eight warps
size_t bulk_slot_bytes();
cudaError_t launch_bulk_gemm(const UmmaPlan *plan, const BulkArgs &a, int epi, int n_sms, int pdl, cudaStream_t st);
// pan = x * gain as a pair, ss[r] = sum x^2; one row per block
cudaError_t launch_norm_pair(const float *x, const void *gain, float *ss, void *pan, int pan_rows, int R, int d, int pdl, cudaStream_t st);
// kv_len[sequence] += rows for every segment
cudaError_t launch_advance(int32_t *kv_len, const RowSegs &segs, int nseg, cudaStream_t st);

// ---- up to 64 rows: chained projections with one writer per output (k_cluster.cu); d, qd, f multiples of 128, kvd and vocab of 16
// The width the kernel is built for at most (64 activation rows high and low are one MMA operand of 128).  One step of 7B against the
// chained launch it replaces: 1 row over 512 keys 2612 us, 2803; 16 over 803 2718, 3235; 2 x 16 3024, 4079; 4 x 16 over 2048 4615, 4882.
constexpr int kClusterRows = 64;
constexpr int kClusterSlots = 160;                   // CTAs that the slots of the row sums of squares are laid out for
struct ClusterModel {
  int n_layers, d, qd, kvd, f, vocab;
  const void *const *wq, *const *wk, *const *wv, *const *wo, *const *w_gate, *const *w_up, *const *w_down, *lm_head;   // host arrays of device pointers
};
struct ClusterPlan;
bool cluster_shape_ok(int d, int qd, int kvd, int f, int vocab);
cudaError_t cluster_plan_create(const ClusterModel &m, void *pan_x, void *pan_a, void *pan_h, ClusterPlan **out);
void cluster_plan_destroy(ClusterPlan *p);
// Against the chained launch; false without a plan.  fused: that launch would have the fused attention in front of it.
bool cluster_pays(const ClusterPlan *pl, int R, int max_len, bool fused);
struct ClusterArgs {
  int R;
  float *x, *qkv;                 // [R, d] residual, [R, qd + 2 kvd] (lacking 1/rms)
  void *pan_x, *pan_h;            // operand pairs
  const void *g_ffn, *g_next;     // gains behind the O and the down projection of this launch
  float *ss_x, *ss_ffn;           // [kClusterSlots][kClusterRows]
  float *ss_attn;                 // [R], written by the QKV projection
  float eps;
  unsigned int *bar;              // [8 * n_layers + 2], zero when a forward starts
  int withheld;                   // test aid: arrivals that the launch's grid barriers wait for and nobody makes
  const int32_t *tokens, *perm; float beta; unsigned long long *amax; float *logits;
  unsigned int *err;
};
// projections [first, last), four at most, one after the other: 4 * layer + {0 QKV, 1 O, 2 gate/up, 3 down}, 4 * n_layers: the LM head
cudaError_t launch_cluster_chain(const ClusterPlan *pl, const ClusterArgs &a, int first, int last, int pdl, cudaStream_t st);
// x = E[token], pan = x * gain as a pair, ss[r] = sum x^2; words[0 .. n_words) = 0
cudaError_t launch_embed_pair(const int32_t *tokens, const void *emb, const void *gain, float *x, void *pan, float *ss, unsigned int *words, int n_words,
                              int R, int d, int pdl, cudaStream_t st);

// Up to four projections in one launch, each consuming the previous one's reduced output; bar: n-1 zeroed words.
// bar_b: n zeroed words (panel-ready barriers), needed when the rows exceed 16 and the plans have panels.
// sync (optional, used up to 16 rows): how each projection is tied to the others, instead of a grid barrier
// after every one.  wait_bar / sig_bar: index of the grid barrier (word of `bar`) the projection waits on before
// its first activation load / arrives on when done, -1 for none.  td_prod: the projection is claimed tile by tile
// and counts finished chunks per 128-column output tile in counter set td_prod (several projections may feed one
// set: partial sums of the same output); td_cons: it is claimed k range by k range and stages a k-block once the
// tile of set td_cons it reads is complete.  tile_done: zeroed words, td_stride per counter set.
// epi_bar: grid barrier the projection's epilogue warps pass before their first reduction into the output (-1: none);
// needed when the output buffer is still being read by a projection that this one does not otherwise wait for.
struct ChainSync { int wait_bar, sig_bar, td_prod, td_cons, epi_bar; };
constexpr int kChainMax = 6;     // projections in one chained launch
cudaError_t launch_gemm_chain(const UmmaPlan *const *plans, const GemmArgs *args, int n, unsigned int *bar,
                              unsigned int *claim, unsigned int *bar_b, const ChainSync *sync, unsigned int *tile_done,
                              int td_stride, const ZeroList *zero, int pdl, cudaStream_t st, int cta_pairs = 0);

}  // namespace fc
