// Internal declarations shared by the kernels and the C-ABI layer of libcmsd.so.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace cmsd {

// The streaming kernel runs as few, large CTAs (one per SM): warps of one CTA
// are scheduled evenly, warps of co-resident CTAs are not.  512 threads of 128
// registers, four vectors per tensor and stage: B=256 K=16 V=152064 bf16 takes
// 382 us a sampled call against 395 us with 768 threads and two (402 us with the
// loop that had conditions and copies in it), 480 and 448 threads 388 and 397
// us, two CTAs of 256 threads 389 us.  Short rows that warps cross the ends of
// take 768 threads and two vectors (stream_threads in cmsd_api.cu).
constexpr int kStreamThreads = 512;
constexpr int kStreamThreadsShort = 768;
__host__ __device__ constexpr int stream_unroll(int threads) { return threads > kStreamThreads ? 2 : 4; }
#ifndef CMSD_RES_THREADS
#define CMSD_RES_THREADS 256
#endif
constexpr int kResThreads = CMSD_RES_THREADS;   // threads per CTA of the resample kernel
constexpr int kResWarps = kResThreads / 32;
constexpr int kStreamWarps = kStreamThreads / 32;
constexpr int kMaxWarpsPerSM = 64;            // 2048 threads / SM
constexpr int kMaxRaggedB = 12000;            // B limit when k_row is given (prefix in smem)
constexpr int kPackedMaxK = 16;               // windows merged through one 64-bit counter

enum Mode { kModeConf = 0, kModeVerify = 1, kModeFused = 2 };

// Second pass over one row of a sequence, after its first-reject scan:
// the residual draw at a rejected position (sampled rule), or the token of
// the verifier's extra row when every draft was accepted (bonus row).
enum SeqKind { kSeqNone = 0, kSeqResidual = 1, kSeqBonus = 2 };

// Residual / bonus races run over groups of kGroup consecutive entries.
constexpr int kGroup = 32;

// dynamic shared memory of one streaming CTA: the k_row prefix (ragged windows)
__host__ __device__ inline size_t stream_smem_bytes(int B, bool ragged) {
  return ragged ? (((size_t)(B + 1) * sizeof(int) + 127) / 128) * 128 : 0;
}

// One warp's reduction over one row segment (or, in the row merge, the
// reduction over all segments).  Drafter: running max m, s = sum e^(z-m),
// t2 = sum e^(z-m) (z-m) log2(e), second largest logit, lowest argmax.
// Target: running max, s = sum e^(z-m), lowest argmax, count of logits
// strictly above the drafted token's (saturating at beta_rank).
struct __align__(16) Partial {
  float d_m, d_s, d_t2, d_top2;
  int d_idx;
  float t_m, t_s;
  int t_idx, t_cnt;
  int pad[3];
};

// One resample warp's result for one queued row: its least race key (or, for
// the bonus argmax, minus its largest logit), its group and its token.
struct __align__(16) UnitResult {
  float key;
  float ref;   // bonus race: the warp's exponent reference (max * log2 e)
  int grp;
  int tok;
};

struct Workspace {
  // counters (zero at rest; each call returns them to zero)
  unsigned* err;                  // [1]   sticky device-side errors
  int* row_done;                  // [B*K] logits of the row already reduced
  unsigned long long* seq_word;   // [B]   K <= 16: rows merged | accept bits | sum of C (fixed point)
  int* seq_done;                  // [B]   K > 16: rows merged
  int* rec_count;                 // [1]   sequences queued for the second pass
  int* res_cta_done;              // [1]   CTAs of the resample kernel that finished
  int* res_done;                  // [B]   groups of each queued row already raced
  // per-call scratch
  int4* rec;                      // [B]   queued rows: (b, position, kind, 0)
  unsigned long long* row_conf;   // [B*K] C of each position, fixed point C * 2^36
  int* row_acc;                   // [B*K] accept bit (K > 16 epilogue)
  float2* row_dstat;              // [B*K] drafter (max * log2e, sum e^(z-max))
  float2* row_tstat;              // [B*K] target  (the same)
  Partial* part;                  // [B*K + warps]
  UnitResult* rpart;              // [B + warps]
};

// Fewest logits per warp slice: small problems are cut finely (latency), large
// rows into at most about 128 pieces (each piece costs one partial to merge).
// Measured on one-call latencies: 1024 beat 2048 by 2-3 us at B=1 K=4
// V=32000, and 512 or 256 gained nothing more.
__host__ __device__ inline int64_t stream_min_len(int V) {
  const int64_t a = (int64_t)V / 128 + 64;
  return a > 1024 ? a : 1024;
}
// a / b for 0 <= a, 0 < b, in 32-bit arithmetic when both fit.
__host__ __device__ inline int64_t div_nn(int64_t a, int64_t b) {
  if (a <= 0x7FFFFFFF && b <= 0x7FFFFFFF) return (int64_t)((uint32_t)a / (uint32_t)b);
  return a / b;
}

// How the present-row stream (R rows of V logits, N = R*V elements) is cut
// into warp slices.  When there are at least as many warps as rows, each row
// is cut into wpr pieces of one warp each (no slice crosses a row end, so
// every warp streams one segment); otherwise the stream is cut into W equal
// runs of 128-byte lines.  Slices start on multiples of 128 bytes from the
// row (or stream) start, so that a warp's 512-byte loads cover whole 32-byte
// sectors when the rows themselves are 128-byte aligned; a 16-byte offset
// would make every load touch one sector more (the last slice ends at N).
// Formed on the host for full windows: its 64-bit divisions kept a slice's
// first loads waiting (0.4 us of a 11.2 us call at B=64 K=1 V=128256).
constexpr int kLineVecs = 8;   // 16-byte vectors per 128-byte line
struct StreamSplit {
  StreamSplit() = default;
  int64_t N;
  int W;          // warps with work
  int V, VEC;
  int wpr;        // > 0: row-aligned split with wpr warps per row
  int qv, rv;     // row-aligned: V / wpr, V % wpr
  int64_t q;      // flat: vectors per warp (the first rem warps one more)
  int rem;
  __host__ __device__ StreamSplit(int R, int V_, int vec, int nwarps, int64_t min_len) {
    V = V_;
    VEC = vec;
    N = (int64_t)R * V;
    int64_t want = div_nn(N, min_len);
    if (want < 1) want = 1;
    const int Wmax = (int)(want < nwarps ? want : nwarps);
    int p = nwarps / R;                              // pieces per row that fit
    const int pm = (int)div_nn(V, min_len);
    const int pmax = pm > 0 ? pm : 1;
    if (p > pmax) p = pmax;
    if (p >= 1 && (int64_t)p * R * 4 >= (int64_t)Wmax * 3) {   // uses at least 3/4 of the warps
      wpr = p;
      W = p * R;
      qv = V / p;
      rv = V - qv * p;
      q = 0;
      rem = 0;
    } else {
      wpr = 0;
      W = Wmax;
      qv = rv = 0;
      const int64_t nv = N / (VEC * kLineVecs);
      q = div_nn(nv, W);
      rem = (int)(nv - q * W);
    }
  }
  __host__ __device__ int64_t start(int w) const {
    if (w >= W) return N;
    if (wpr > 0) {
      const int row = w / wpr, k = w - row * wpr;
      const int off = k * qv + (k < rv ? k : rv);
      return (int64_t)row * V + (off & ~(VEC * kLineVecs - 1));
    }
    return ((int64_t)w * q + (w < rem ? w : rem)) * VEC * kLineVecs;
  }
  // warps holding the first and the last element of row ar
  __host__ __device__ int first_warp(int ar) const { return wpr > 0 ? ar * wpr : owner_flat((int64_t)ar * V); }
  __host__ __device__ int last_warp(int ar) const {
    return wpr > 0 ? ar * wpr + wpr - 1 : owner_flat((int64_t)ar * V + V - 1);
  }
  __host__ __device__ int owner_flat(int64_t e) const {
    const int64_t ev = e / (VEC * kLineVecs);
    const int64_t big = (q + 1) * rem;
    const int w = ev < big ? (int)div_nn(ev, q + 1) : rem + (int)div_nn(ev - big, q);
    return w < W ? w : W - 1;
  }
};

struct StreamArgs {
  const void* draft;
  const void* target;
  const int* tokens;
  const int* k_row;
  int B, K, V;
  int Kt;                 // verifier rows per sequence: K, or K + 1 with the bonus row
  int Ko;                 // out_tokens columns: K, or K + 1 with the bonus row
  int k_min, k_max, k_fixed;
  float lam0, lam1, lam2, beta_sig;
  float inv_log_v;        // 1 / ln V
  float soft_norm;        // 1 / (1 - 1/V)
  int beta_rank;
  float alpha, tau_base, gamma;
  int tau_sign;
  int bonus;
  unsigned long long seed;
  unsigned iteration;
  const float* conf_in;   // verify-only
  const float* lse_in;    // verify-only, SAMPLED
  float* H;
  float* margin;
  int* argmax;
  float* conf;
  float* lse;
  int* k_next;
  int* n_accept;
  int* out_tokens;
  unsigned char* accept;
  Workspace ws;
  int nwarps;             // warps launched
  StreamSplit split;      // full windows: the cut of the B*K rows
  int rec_by_seq;         // 1: second-pass records at each sequence's own slot rec[b], every sequence
                          // writing one (the draw by group bounds); 0: a compacted queue (rec_count)
};

// Kernel launchers (one translation unit per dtype).  `second`: this call
// queues rows for the resample kernel (sampled rule or bonus row).
// threads: kStreamThreads or kStreamThreadsShort.
cudaError_t launch_stream_f32(int mode, bool sampled, bool second, const StreamArgs& a, int grid, int threads,
                              size_t smem, cudaStream_t s);
cudaError_t launch_stream_bf16(int mode, bool sampled, bool second, const StreamArgs& a, int grid, int threads,
                               size_t smem, cudaStream_t s);
// The pass in one launch, a cluster of nc CTAs of `threads` (256 or 512)
// threads per sequence (cmsd_seq_impl.cuh).
cudaError_t launch_seq_f32(int mode, bool sampled, bool second, const StreamArgs& a, int nc, int threads,
                            cudaStream_t s);
cudaError_t launch_seq_bf16(int mode, bool sampled, bool second, const StreamArgs& a, int nc, int threads,
                            cudaStream_t s);
// Clusters of nc such CTAs that can be resident on the current device (0: none).
int seq_clusters_f32(int nc, int threads);
int seq_clusters_bf16(int nc, int threads);
bool seq_draw_fits(int dtype, int V);
cudaError_t launch_resample_f32(bool sampled, const StreamArgs& a, int grid, cudaStream_t s);
cudaError_t launch_resample_bf16(bool sampled, const StreamArgs& a, int grid, cudaStream_t s);
// The draw by group bounds (residual and bonus tokens): clusters of nc CTAs,
// one sequence per cluster at a time; draw_clusters says how many such
// clusters can be resident on the current device for rows of V entries (0:
// resample_kernel takes the call).
cudaError_t launch_draw_f32(bool sampled, const StreamArgs& a, int clusters, int nc, cudaStream_t s);
cudaError_t launch_draw_bf16(bool sampled, const StreamArgs& a, int clusters, int nc, cudaStream_t s);
int draw_clusters_f32(int V, int nc);
int draw_clusters_bf16(int V, int nc);
// The residual draw with its share staged in shared memory (clusters of a
// fixed size); how many clusters can be resident (0: the share does not fit).
cudaError_t launch_resample_bound_f32(const StreamArgs& a, int clusters, cudaStream_t s);
cudaError_t launch_resample_bound_bf16(const StreamArgs& a, int clusters, cudaStream_t s);
int resample_bound_clusters_f32(int V);
int resample_bound_clusters_bf16(int V);
cudaError_t occupancy_stream(int dtype, int mode, bool sampled, bool second, int threads, size_t smem,
                             int* blocks_per_sm);
cudaError_t occupancy_resample(int dtype, bool sampled, int* blocks_per_sm);
cudaError_t launch_philox_fill(unsigned long long seed, uint32_t c0, uint32_t c1, uint32_t c2,
                               uint32_t c3, uint32_t* out, size_t n, cudaStream_t s);

// The drafter's LM head fused with its confidence signals (cmsd_lmhead.cu).
struct LmHeadArgs {
  const uint16_t* hidden;        // bf16 [R][d]
  const uint16_t* weight;        // bf16 [V][d]
  int R, d, V;
  int nb;                        // hidden rows per block (lmhead_block_rows(R))
  int nct;                       // CTAs per block (each owns a run of the vocabulary)
  float* logits;                 // nullable: f32 [R][V]
  Partial* part;                 // [ceil(R / nb)][nct][nb] per-CTA row statistics
  unsigned* err;                 // error word (bit 2: a wait for a load gave up)
};
int lmhead_block_rows(int R);
int lmhead_ctas_per_block(int sms, int R, int V);
// The GEMM + statistics kernel, then the per-row merge (a programmatic
// dependent on the same stream).  a carries the parameters, the output
// pointers and a workspace with row_conf [R].
cudaError_t launch_lmhead(const LmHeadArgs& h, const StreamArgs& a, cudaStream_t s);

// Host-side checks shared by the entry points (cmsd_api.cu).
int validate_fused(const void* draft_logits, const void* target_logits, const int32_t* draft_tokens,
                   const int32_t* k_row, int B, int K, int V, int dtype, const void* params,
                   const int32_t* n_accept, const int32_t* out_tokens);

}  // namespace cmsd
