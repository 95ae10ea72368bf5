// The drafter's LM head fused with its confidence signals (include/cmsd.h,
// cmsd_lmhead_confidence).
//
// The paper's estimator sits on the drafter's output logits (Sec. I), the
// product z = h W^T of the drafter's last hidden state with its LM-head
// weight, and reads from each logit row the entropy, logit margin and softmax
// margin of Sec. III.B(1).  Here the product runs on the 5th-generation
// tensor cores (tcgen05.mma, bf16 in, fp32 accumulators in tensor memory) and
// each finished tile of 128 vocabulary entries is folded, in the GEMM's
// epilogue, into per-row running statistics: running maximum and
// its first index, second largest logit, and compensated sums of e^(z - ref)
// and e^(z - ref)(z - ref) log2 e against a lazily moved exponent reference
// (the same arithmetic as the logits pass).  The logits never reach HBM
// unless the caller asks for them.  A second small kernel merges the per-CTA
// statistics of each row and computes H, margin, C and the log-sum-exp with
// the logits pass's row arithmetic.
//
// Layout: hidden [R][d] and weight [V][d] row-major bf16 (the usual
// [out][in] layout of a linear layer's weight), d a multiple of 64.  Each CTA
// owns a contiguous run of the vocabulary for one block of hidden rows and
// streams its weight rows once through a ring of shared-memory stages filled
// by 2D tensor-memory-access (TMA) loads: per stage one box of 64 hidden
// dimensions x 128 weight rows and the same dimensions of the hidden rows, both
// with the 128-byte swizzle that the MMA's shared-memory descriptors name; rows
// past R or V arrive as zeros.  The hidden block is re-read from L2 for every
// tile.
//
// Bounds, on a GB300: up to 128 hidden rows DRAM (R=64 d=2048 V=128256: 525.6 MB
// in 90.4 us, 5.8 TB/s); at 256 rows the MMAs, whose operands take the shared
// memory's bandwidth (108 us, 1.25 PFLOP/s; 131 us when the epilogue transposed
// every tile); small calls the launch, the fill of the ring, the hidden rows,
// which every CTA reads from the same lines of L2 (R=1 d=1024 V=32000 17.3 us,
// R=16 20.2), and the merge kernel.
#include <cuda.h>

#include <mutex>

#include "cmsd_stream_impl.cuh"

namespace cmsd {
namespace {

constexpr int kMergeRowsPerCta = 8;                 // one warp per row

// ---- shared-memory barriers and 2D TMA loads -----------------------------------
// box of the 2D tensor map at (x, y) (x: innermost, in elements) into shared
// memory at dst, completing `bar` by transaction count
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, int x, int y, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::
          "r"(dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(bar)
      : "memory");
}

// The vocabulary run of CTA `cta` of a row block: nct near-equal runs of
// 8 entries ([v0, v1), v1 <= V).
__device__ __forceinline__ void cta_run(int V, int nct, int cta, int& v0, int& v1) {
  const int n8 = (V + 7) / 8;
  const int q = n8 / nct, rem = n8 - q * nct;
  v0 = (cta * q + (cta < rem ? cta : rem)) * 8;
  const int e = ((cta + 1) * q + (cta + 1 < rem ? cta + 1 : rem)) * 8;
  v1 = e < V ? e : V;
}

// Fold 32 consecutive logits (vocabulary entries v0 .. v0+31, those at or
// past vend masked) into a thread's running drafter statistics.
__device__ __forceinline__ void fold32(DLane& st, float (&z)[32], int v0, int vend) {
  if (v0 + 32 > vend) {
#pragma unroll
    for (int k = 0; k < 32; ++k)
      if (v0 + k >= vend) z[k] = -pos_inf();
  }
  // top-2 of the 32 in four independent chains, then with the lane's so far
  float a1[4], a2[4];
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    a1[c] = z[8 * c];
    a2[c] = kNegInit;
#pragma unroll
    for (int k = 1; k < 8; ++k) {
      a2[c] = fmaxf(a2[c], fminf(a1[c], z[8 * c + k]));
      a1[c] = fmaxf(a1[c], z[8 * c + k]);
    }
  }
#pragma unroll
  for (int o = 2; o; o >>= 1) {
#pragma unroll
    for (int c = 0; c < o; ++c) {
      a2[c] = fmaxf(fmaxf(a2[c], a2[c + o]), fminf(a1[c], a1[c + o]));
      a1[c] = fmaxf(a1[c], a1[c + o]);
    }
  }
  st.f2 = fmaxf(fmaxf(st.f2, a2[0]), fminf(st.f1, a1[0]));
  st.f1 = fmaxf(st.f1, a1[0]);
  // entries come in increasing index order, so a strict increase keeps the
  // lowest index; the first entry equal to the new maximum is its index
  if (a1[0] > st.m) {
    int k0 = 0;
#pragma unroll
    for (int k = 31; k >= 0; --k) k0 = z[k] == a1[0] ? k : k0;
    st.pos = v0 + k0;
    st.m = a1[0];
  }
  // one reference check, then the exponentials, summed among themselves
  const float me = d_mexp(st);
  if (me > st.ref + kRefSlack) d_reref(st, me);
  const float nc = neg_clamp();
  const u64 L = dup2(kLog2e);
  u64 ss = 0ull, ts = 0ull;
#pragma unroll
  for (int k = 0; k < 16; ++k) {
    const u64 x = fma2(pack2(fmaxf(z[2 * k], nc), fmaxf(z[2 * k + 1], nc)), L, st.negrL);
    const u64 e = ex2_2(x);
    ss = add2(ss, e);
    ts = fma2(e, x, ts);
  }
  kahan(st.s, st.cs, lo32f(ss) + hi32f(ss));
  kahan(st.t, st.ct, lo32f(ts) + hi32f(ts));
}

// ===========================================================================
// the product on the 5th-generation tensor cores, the statistics in its epilogue
// ===========================================================================
//
// The MMA's M is the hidden rows and its N the vocabulary, so a TMEM lane is a
// hidden row and its columns are consecutive logits of that row: an epilogue
// thread reads and folds its own row, without a transpose.  (With the
// vocabulary as M every chunk went through shared memory behind two barriers,
// folded by four warps: at 256 rows a tile took 17 us to fold against 11 us of
// MMAs.)  A tile is 128 vocabulary entries.  Blocks of H = 64, 128 or 256
// hidden rows: 64 rows fill the 128 lanes twice over, 256 rows take two MMAs
// and accumulators of 128 lanes.
//
// One CTA of 320 threads per SM:
//   warp 0      lane 0 issues the TMA loads of each stage (weight box of 64 x
//               128 rows = the MMA's B, hidden boxes = its A);
//   warp 1      allocates TMEM (two sets of accumulators of 128 columns), and
//               lane 0 issues tcgen05.mma (K = 16 per instruction) and the
//               commits;
//   warps 2..9  the epilogue: warp w reads TMEM lanes 32 (w mod 4) ..; the two
//               warps of a lane quarter, and the two copies of 64 rows, take
//               an equal part of the tile's columns each.
// Barriers: full[s] / empty[s] per stage (TMA -> MMA -> TMA), tfull[b] /
// tempty[b] per accumulator set (MMA -> epilogue -> MMA).  Every wait is
// bounded; TMEM is released after the last commit and the last load have
// completed.
constexpr int kTcN = 128;                           // vocabulary entries per tile (MMA N)
constexpr int kTcWStage = kTcN * 128;               // 16 KB: 128 weight rows x 64 bf16
constexpr int kTcEpiThreads = 256;
constexpr int kTcThreads = 64 + kTcEpiThreads;

template <int H>
struct TcShape {
  static_assert(H == 64 || H == 128 || H == 256, "block rows");
  static constexpr int kAcc = H == 256 ? 2 : 1;     // accumulators of 128 lanes
  static constexpr int kSplit = 256 / H;            // threads per hidden row
  static constexpr int kCols = kTcN / kSplit;       // columns each of them folds
  static constexpr int kStages = H == 256 ? 4 : 6;
  static constexpr int kHStage = kAcc * 128 * 128;  // bytes of hidden rows per stage
  static constexpr int kTmem = 2 * kAcc * kTcN;     // TMEM columns
  static constexpr size_t kStageBytes = (size_t)kStages * (kTcWStage + kHStage);
  static constexpr size_t kRedBytes = (size_t)kTcEpiThreads * 20;   // DRed per thread, 5 arrays
  static constexpr size_t kSmem = 1024 + kStageBytes + kRedBytes + 8 * (2 * kStages + 4) + 16;
  static_assert(kSmem <= 227 * 1024, "shared memory");
};
// instruction descriptor, kind::f16: fp32 accumulator, bf16 A and B, both
// K-major, N >> 3 at bit 17, M >> 4 at bit 24
constexpr uint32_t kTcIdesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(kTcN >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);

// Shared-memory matrix descriptor of a K-major tile with 128-byte rows and the
// 128-byte swizzle: start address, leading offset (unused for this layout),
// stride between 8-row groups = 1024 bytes, descriptor version 1, layout
// SWIZZLE_128B.
__device__ __forceinline__ uint64_t umma_desc_sw128(uint32_t saddr) {
  return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)1 << 16) | ((uint64_t)(1024 >> 4) << 32) |
         ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}

__device__ __forceinline__ void tc_mma(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                       uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(d_tmem),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}
__device__ __forceinline__ void tc_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
// 32 lanes x 32 columns of fp32 from TMEM: thread i gets lane (taddr lane + i), columns c .. c + 31
__device__ __forceinline__ void tc_ld32(uint32_t taddr, float (&v)[32]) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
      "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr)
      : "memory");
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int k = 0; k < 32; ++k) v[k] = __uint_as_float(r[k]);
}
// named barrier among the epilogue threads (barrier 0 is __syncthreads)
__device__ __forceinline__ void epi_bar() { asm volatile("bar.sync 1, 256;" ::: "memory"); }

// hrows: rows loaded of a block (lanes beyond them hold whatever was there: a
// lane's result depends on its own row alone).
// tmap_w0, tmap_w1: the weight in boxes of the rows of a run's last tile (runs
// of q and q + 1 groups of eight entries), so that no row is read twice (a
// whole box there made the kernel read 1.06 x the weight at V=128256).
template <int H>
__global__ void __launch_bounds__(kTcThreads, 1) lmhead_tc_kernel(const LmHeadArgs h, const int hrows, const int tail0,
                                                                 const int tail1,
                                                                 const __grid_constant__ CUtensorMap tmap_h,
                                                                 const __grid_constant__ CUtensorMap tmap_w,
                                                                 const __grid_constant__ CUtensorMap tmap_w0,
                                                                 const __grid_constant__ CUtensorMap tmap_w1) {
  using S = TcShape<H>;
  constexpr int kStages = S::kStages;
  extern __shared__ __align__(1024) unsigned char tc_smem_raw[];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int rb = blockIdx.x / h.nct, cta = blockIdx.x - rb * h.nct;
  int v0, v1;
  cta_run(h.V, h.nct, cta, v0, v1);
  const int ntiles = v1 > v0 ? (v1 - v0 + kTcN - 1) / kTcN : 0;
  // the last tile's rows: runs of q + 1 groups come first
  const int n8 = (h.V + 7) / 8;
  const bool longer = cta < n8 - (n8 / h.nct) * h.nct;
  const CUtensorMap* map_last = longer ? &tmap_w1 : &tmap_w0;
  const int tail = longer ? tail1 : tail0;
  const int nkc = h.d / 64;
  const int G = ntiles * nkc;
  const int row0 = rb * H;

  const uint32_t raw = smem_u32(tc_smem_raw);
  const uint32_t pad = ((raw + 1023u) & ~1023u) - raw;
  unsigned char* sm = tc_smem_raw + pad;
  const uint32_t sW = raw + pad, sH = sW + kStages * kTcWStage;
  float* s_red = reinterpret_cast<float*>(sm + S::kStageBytes);
  const uint32_t bars = smem_u32(sm + S::kStageBytes + S::kRedBytes);
  const uint32_t full = bars, empty = bars + 8 * kStages;
  const uint32_t tfull = bars + 16 * kStages, tempty = tfull + 16;
  uint32_t* s_taddr = reinterpret_cast<uint32_t*>(sm + S::kStageBytes + S::kRedBytes + 8 * (2 * kStages + 4));
  if (tid == 0) {
    for (int k = 0; k < kStages; ++k) {
      mbar_init(full + 8 * k, 1);
      mbar_init(empty + 8 * k, 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(tfull + 8 * b, 1);
      mbar_init(tempty + 8 * b, kTcEpiThreads);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(s_taddr)),
                 "r"(S::kTmem)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  // everything above overlaps the end of what precedes this grid on the stream
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  tc_fence_after();
  const uint32_t tbase = *s_taddr;
  bool ok = true;

  if (warp == 0) {
    // ---- producer ----------------------------------------------------------
    if (lane == 0) {
      for (int g = 0; g < G; ++g) {
        const int slot = g % kStages;
        if (g >= kStages && ok) ok = mbar_wait(empty + 8 * slot, (uint32_t)((g / kStages - 1) & 1));
        const int t = g / nkc, kc = g - t * nkc;
        const bool last = t == ntiles - 1;
        mbar_arrive_tx(full + 8 * slot, (last ? tail * 128 : kTcWStage) + (H == 64 ? 2 : 1) * hrows * 128);
        tma_load_2d(sW + slot * kTcWStage, last ? map_last : &tmap_w, kc * 64, v0 + t * kTcN, full + 8 * slot);
        const uint32_t hdst = sH + slot * S::kHStage;
#pragma unroll
        for (int c = 0; c < (H == 64 ? 2 : 1); ++c)       // the hidden rows (64 of them: twice)
          tma_load_2d(hdst + c * 64 * 128, &tmap_h, kc * 64, row0, full + 8 * slot);
      }
    }
  } else if (warp == 1) {
    // ---- MMA issuer --------------------------------------------------------
    if (lane == 0) {
      for (int t = 0; t < ntiles; ++t) {
        const int b = t & 1;
        if (t >= 2 && ok) ok = mbar_wait(tempty + 8 * b, (uint32_t)((t / 2 - 1) & 1));
        tc_fence_after();
        const uint32_t d = tbase + (uint32_t)(b * S::kAcc * kTcN);
        for (int kc = 0; kc < nkc; ++kc) {
          const int g = t * nkc + kc, slot = g % kStages;
          if (ok) ok = mbar_wait(full + 8 * slot, (uint32_t)((g / kStages) & 1));
          tc_fence_after();
          const uint64_t wd = umma_desc_sw128(sW + slot * kTcWStage);
#pragma unroll
          for (int c = 0; c < S::kAcc; ++c) {
            const uint64_t hd = umma_desc_sw128(sH + slot * S::kHStage + c * 128 * 128);
#pragma unroll
            for (int ks = 0; ks < 4; ++ks)        // K = 16 per instruction: 32 bytes along the row
              tc_mma(d + c * kTcN, hd + (uint64_t)(2 * ks), wd + (uint64_t)(2 * ks), kTcIdesc, (kc | ks) != 0);
          }
          // the stage may be refilled once these MMAs are done
          tc_commit(empty + 8 * slot);
        }
        tc_commit(tfull + 8 * b);                  // the accumulator is complete
      }
    }
    __syncwarp();
  } else {
    // ---- epilogue: warps 2..9 ------------------------------------------------
    const int e = tid - 64;                        // 0 .. 255
    const int q = warp & 3;                        // TMEM lane quarter this warp may read
    const int m = q * 32 + lane;                   // its TMEM lane
    const int grp = (warp - 2) >> 2;               // the two warps of a quarter
    const int acc = H == 256 ? grp : 0;
    const int row = H == 256 ? grp * 128 + m : (H == 128 ? m : (m & 63));      // hidden row within the block
    const int part = H == 256 ? 0 : (H == 128 ? grp : ((m >> 6) * 2 + grp));   // its part of the columns
    DLane st;
    dlane_init(st);
    for (int t = 0; t < ntiles; ++t) {
      const int b = t & 1;
      if (ok) ok = mbar_wait(tfull + 8 * b, (uint32_t)((t / 2) & 1));
      __syncwarp();
      tc_fence_after();
      const uint32_t src = tbase + ((uint32_t)(q * 32) << 16) + (uint32_t)((b * S::kAcc + acc) * kTcN + part * S::kCols);
      const int vq = v0 + t * kTcN + part * S::kCols;
#pragma unroll 1
      for (int c = 0; c < S::kCols; c += 32) {
        float z[32];
        __syncwarp();                              // (the fold below may have diverged)
        tc_ld32(src + c, z);
        if (c + 32 == S::kCols) {
          tc_fence_before();
          mbar_arrive(tempty + 8 * b);             // this thread's columns have been read
        }
        if (h.logits && row0 + row < h.R) {
          float* dst = h.logits + (size_t)(row0 + row) * h.V + vq + c;
#pragma unroll
          for (int k = 0; k < 32; ++k)
            if (vq + c + k < v1) dst[k] = z[k];
        }
        fold32(st, z, vq + c, v1);
      }
    }
    float fs, ft2;
    d_final(st, fs, ft2);
    DRed x{d_mexp(st), fs, ft2, st.f2, st.pos};
    if (S::kSplit > 1) {                           // the threads of a row: part 0 merges the others'
      if (part > 0) {
        s_red[e] = x.m;
        s_red[kTcEpiThreads + e] = x.s;
        s_red[2 * kTcEpiThreads + e] = x.t2;
        s_red[3 * kTcEpiThreads + e] = x.top2;
        s_red[4 * kTcEpiThreads + e] = __int_as_float(x.idx);
      }
      epi_bar();
      if (part == 0) {
#pragma unroll
        for (int c = 1; c < S::kSplit; ++c) {
          // the epilogue thread of this row's part c: warp group c & 1, the other copy of 64 rows for c > 1
          const int mo = H == 64 && (c >> 1) ? m + 64 : m;
          const int eo = 32 * (((c & 1) << 2) + (((mo >> 5) + 2) & 3)) + lane;
          fold_d(x, DRed{s_red[eo], s_red[kTcEpiThreads + eo], s_red[2 * kTcEpiThreads + eo],
                         s_red[3 * kTcEpiThreads + eo], __float_as_int(s_red[4 * kTcEpiThreads + eo])});
        }
      }
    }
    if (part == 0) {
      Partial p;
      p.d_m = x.m; p.d_s = x.s; p.d_t2 = x.t2; p.d_top2 = x.top2; p.d_idx = x.idx;
      p.t_m = 0.f; p.t_s = 0.f; p.t_idx = 0; p.t_cnt = 0;
      p.pad[0] = p.pad[1] = p.pad[2] = 0;
      h.part[((size_t)rb * h.nct + cta) * H + row] = p;
    }
  }
  if (!ok) atomicOr(h.err, 4u);
  // teardown: the MMA issuer's last commit covers every MMA of the CTA; then
  // every thread is past its last TMEM access and TMEM is released
  if (warp == 1 && lane == 0 && ntiles > 0) {
    const int t = ntiles - 1;
    if (!mbar_wait(tfull + 8 * (t & 1), (uint32_t)((t / 2) & 1))) atomicOr(h.err, 4u);
  }
  if (warp == 0 && lane == 0) {                    // no TMA box still in flight into this CTA
    for (int g = (G > kStages ? G - kStages : 0); g < G; ++g)
      if (!mbar_wait(full + 8 * (g % kStages), (uint32_t)((g / kStages) & 1))) atomicOr(h.err, 4u);
  }
  __syncwarp();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tbase), "r"(S::kTmem) : "memory");
}

// One warp per hidden row: fold the row's per-CTA partials, then the row's
// signals and confidence (the logits pass's row arithmetic).
__global__ void __launch_bounds__(32 * kMergeRowsPerCta) lmhead_merge_kernel(const LmHeadArgs h, const StreamArgs a) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");   // (the next call's grid waits for this one's end)
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int lane = threadIdx.x & 31;
  const int r = blockIdx.x * kMergeRowsPerCta + (threadIdx.x >> 5);
  if (r >= h.R) return;                            // whole warps
  const int rb = r / h.nb, row = r - rb * h.nb;
  const Partial* base = h.part + (size_t)rb * h.nct * h.nb + row;
  DRed m = dred_empty();
  constexpr int kBatch = 8;                        // partials in flight per lane
  for (int k0 = lane; k0 < h.nct; k0 += 32 * kBatch) {
    float4 x0[kBatch], x1[kBatch];
#pragma unroll
    for (int j = 0; j < kBatch; ++j) {
      const int k = k0 + 32 * j;
      if (k < h.nct) {
        const float4* src = reinterpret_cast<const float4*>(base + (size_t)k * h.nb);
        x0[j] = __ldcg(src);
        x1[j] = __ldcg(src + 1);
      }
    }
#pragma unroll
    for (int j = 0; j < kBatch; ++j)
      if (k0 + 32 * j < h.nct) fold_d(m, DRed{x0[j].x, x0[j].y, x0[j].z, x0[j].w, __float_as_int(x1[j].x)});
  }
  const DRed dr = reduce_d(m);
  row_results<kModeConf, false>(a, r, 0, 0, dr, tred_empty(), 0.f, 0.f, 0.f, 0.f, lane);
}

}  // namespace

// Hidden rows per block: the least of 64, 128, 256 that holds R (more rows
// than 256 take several blocks, each reading the weight once).
int lmhead_block_rows(int R) { return R <= 64 ? 64 : (R <= 128 ? 128 : 256); }

int lmhead_ctas_per_block(int sms, int R, int V) {
  const int nb = lmhead_block_rows(R);
  const int nrb = (R + nb - 1) / nb;
  int nct = sms / (nrb > 0 ? nrb : 1);
  const int n8 = (V + 7) / 8;
  if (nct > n8) nct = n8;
  return nct < 1 ? 1 : nct;
}

namespace {
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;
  static bool tried = false;
  static std::mutex mu;
  std::lock_guard<std::mutex> lk(mu);
  if (!tried) {
    tried = true;
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = (EncodeTiledFn)p;
  }
  return fn;
}
// a [rows][d] bf16 matrix read in boxes of 64 x box_rows, 128-byte swizzle,
// out-of-range rows read as zeros
bool encode_rows(CUtensorMap* m, const void* base, int d, int rows, int box_rows) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  const cuuint64_t dims[2] = {(cuuint64_t)d, (cuuint64_t)rows};
  const cuuint64_t strides[1] = {(cuuint64_t)d * 2};
  const cuuint32_t box[2] = {64u, (cuuint32_t)box_rows};
  const cuuint32_t estr[2] = {1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}
}  // namespace

template <int H>
cudaError_t launch_tc(const LmHeadArgs& h, cudaStream_t s) {
  static unsigned long long done = 0ull;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const unsigned long long bit = 1ull << (dev & 63);
  if (!(__atomic_load_n(&done, __ATOMIC_ACQUIRE) & bit)) {
    e = cudaFuncSetAttribute(lmhead_tc_kernel<H>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TcShape<H>::kSmem);
    if (e != cudaSuccess) return e;
    __atomic_fetch_or(&done, bit, __ATOMIC_ACQ_REL);
  }
  const int nrb = (h.R + H - 1) / H;
  const int n8 = (h.V + 7) / 8, q = n8 / h.nct;
  const int tail0 = q > 0 ? (8 * q - 1) % kTcN + 1 : 8, tail1 = (8 * q + 7) % kTcN + 1;
  int hrows = nrb == 1 ? (h.R + 7) / 8 * 8 : H;    // whole groups of eight rows
  if (hrows > H) hrows = H;
  CUtensorMap tmap_h, tmap_w, tmap_w0, tmap_w1;
  if (!encode_rows(&tmap_h, h.hidden, h.d, h.R, hrows) || !encode_rows(&tmap_w, h.weight, h.d, h.V, kTcN) ||
      !encode_rows(&tmap_w0, h.weight, h.d, h.V, tail0) || !encode_rows(&tmap_w1, h.weight, h.d, h.V, tail1))
    return cudaErrorInvalidValue;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(nrb * h.nct));
  cfg.blockDim = dim3(kTcThreads);
  cfg.dynamicSmemBytes = TcShape<H>::kSmem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, lmhead_tc_kernel<H>, h, hrows, tail0, tail1, tmap_h, tmap_w, tmap_w0, tmap_w1);
}

// Sharing the hidden rows' loads among the CTAs of a cluster would need loads
// that write several CTAs' shared memory.  They are unsafe in a program on
// several GPUs, which loads this same library, and are not used; they gained
// 1 to 18 per cent (us a call with clusters of four, and without: R=16 d=1024
// V=32000 18.3, 20.2; R=64 d=2048 V=128256 88.0, 90.4; R=128 90.1, 91.1; R=8
// d=512 V=8000 9.4 to 10.3, 11.3).
cudaError_t launch_lmhead(const LmHeadArgs& h, const StreamArgs& a, cudaStream_t s) {
  if (h.nb != lmhead_block_rows(h.R)) return cudaErrorInvalidValue;
  const cudaError_t e = h.nb == 64 ? launch_tc<64>(h, s) : (h.nb == 128 ? launch_tc<128>(h, s) : launch_tc<256>(h, s));
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)((h.R + kMergeRowsPerCta - 1) / kMergeRowsPerCta));
  cfg.blockDim = dim3(32 * kMergeRowsPerCta);
  cfg.dynamicSmemBytes = 0;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, lmhead_merge_kernel, h, a);
}

}  // namespace cmsd
