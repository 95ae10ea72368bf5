// The logits pass in one launch, a thread-block cluster per sequence (sm_103a).
//
// For windows of at most 16 positions and problems too small to fill the
// streaming kernel's grid for long (the rule is choose_seq in cmsd_api.cu).
// There the time is not bandwidth but the chain of dependent steps, and the
// streaming kernel's chain goes through global memory: partials and an
// acquire-release atomic per slice, loads of them by the row's merger, an
// atomic per row, a record word and a second kernel that polls it, each step
// an L2 round trip of about a microsecond.  Here a sequence's rows are cut
// over the warps of one cluster and every hand-over is a store into a peer's
// shared memory and a cluster barrier:
//   stream   each warp reduces its pieces (the streaming kernel's arithmetic)
//            and stores their partials into every CTA;
//   rows     barrier; one warp per row, in every CTA alike, merges its partials
//            and takes the row's decision; every CTA finds the first rejection,
//            CTA 0 writes the outputs;
//   draw     under the sampled rule, or for the bonus row, the cluster draws
//            the token itself: every group of a short share from registers
//            (cluster_race), else the race by group bounds (cluster_draw).
//            Its rows were streamed moments ago and come from L2.
// What can be formed before the preceding grid ends (a full window's first
// piece) is, above griddepcontrol.wait.
//
// us a call, the streaming kernel and its draw against one launch, sampled
// bf16: B=4 K=4 V=32000 16.1, 7.7; B=32 K=8 V=128256 35.7, 30.2; B=64 54.2,
// 52.8, where 256 CTAs stream 262.7 MB at 0.87 of the copy rate (at two CTAs an
// SM 48 of the 152 hold one alone, whose loads in flight do not fill its share;
// issue is active 46 %), and 8 us of rows and draw follow.
#pragma once
#include "cmsd_stream_impl.cuh"

namespace cmsd {

constexpr int kSeqMaxCtas = kDrawMaxCtas;   // CTAs per cluster (16: a non-portable size)
constexpr int kSeqMaxK = kPackedMaxK;    // positions per window
// Vectors per lane, tensor and stage: both tensors under the PAPER rule, under
// the sampled rule (four spill there, and cost more registers than the deeper
// stage gains: B=8 K=8 V=128256 14.9 against 13.4 us, B=16 24.4, 22.6, B=64
// 53.2, 52.8; B=1 12.1, 12.5), and one tensor alone (six or four: verify
// B=128 K=8 V=128256 41.5, 43.9 against 40.9).
#ifndef CMSD_SEQ_UNROLL
#define CMSD_SEQ_UNROLL 4
#endif
#ifndef CMSD_SEQ_UNROLL_S
#define CMSD_SEQ_UNROLL_S 3
#endif
#ifndef CMSD_SEQ_UNROLL1
#define CMSD_SEQ_UNROLL1 8
#endif
// ---------------------------------------------------------------------------
// the kernel
// ---------------------------------------------------------------------------

// The cut of a window of kb rows over the cluster's warps, by kb.
struct SeqSplit {
  int nc;                                // CTAs per cluster
  int part_bytes;                        // shared memory of the partials
  int len[kSeqMaxK + 1];                 // entries per piece
  short pieces[kSeqMaxK + 1];            // pieces per row
};

// Piece u of the window: piece k of row i.
template <typename T>
struct SeqPiece {
  int i, k;
  const T* dp;
  const T* tp;
  Seg sg;
};
template <typename T, int MODE>
__device__ __forceinline__ SeqPiece<T> seq_piece(const StreamArgs& a, const SeqSplit& sp, int b, int u, int p, int len) {
  SeqPiece<T> x;
  x.i = (int)((unsigned)u / (unsigned)p);
  x.k = u - x.i * p;
  x.dp = (const T*)a.draft + ((size_t)b * a.K + x.i) * (size_t)a.V;
  x.tp = MODE != kModeConf ? (const T*)a.target + ((size_t)b * a.Kt + x.i) * (size_t)a.V : nullptr;
  x.sg = seg_geom<T>(MODE != kModeVerify ? x.dp : x.tp, x.k * len, a.V, len);
  return x;
}

// A row's decision as every CTA of the cluster keeps it.
struct __align__(16) SeqRow {
  float4 stat;                           // sampled rule: drafter, then target (max * log2e, sum)
  unsigned long long cfx;
  int acc, pad;
};

// The draw of cluster_draw by racing every group of the share exactly, for
// shares of at most Q blocks of four groups per lane set: each lane set holds
// the vectors of its groups in registers, so the row's two loads, the keys
// and one exchange are the whole chain (cluster_draw: maxima, bounds, probes, an
// exchange, the groups that remain, the exchange).  Against cluster_draw, in
// us a call: B=4 K=8 V=128256 (16 CTAs) 13.8 -> 12.5, B=16 K=4 V=32000 11.4
// -> 10.1, with the bonus row B=8 K=8 V=128256 18.9 -> 14.9 and B=32 (Q = 2)
// 31.8 -> 30.8.  More than eight groups per lane set cost more exponentials
// than the bounds save; so do rows off 16-byte boundaries at Q = 2 (verify
// B=96 K=12 V=32001 ragged: 21.0 against 22.6), which take two loads and a
// shift per vector.
//
// Four groups' sums per block are reduced by exchanging halves (lane bit 0,
// then bit 1), which leaves group k's in the lanes with sub & 3 == k, and
// every sum is formed in the order of group_key.
template <typename T, int NT, int Q>
__device__ __forceinline__ void cluster_race(const StreamArgs& a, cg::cluster_group& cl, int nc, int cr, int b, int pos,
                                             bool bonus, const T* tp, const T* dp, float2 ts, float2 ds,
                                             DrawShared<T, NT>& sh) {
  constexpr int VEC = Elem<T>::kVec;
  constexpr int LPG = DrawShared<T, NT>::kLpg;
  constexpr int SETS = DrawShared<T, NT>::kSets;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int sub = lane % LPG, set = tid / LPG;
  const int ng = (a.V + kGroup - 1) / kGroup;
  const int ngs = draw_share(ng, nc);
  const int gs = cr * ngs;                                   // the share: groups [gs, gs + nloc)
  const int nloc = max(0, min(ng, gs + ngs) - gs);
  const uint32_t k0 = seed_lo(a.seed), k1 = seed_hi(a.seed);
  const uint32_t cw_grp = iter_word(a.iteration, kPurposeGroup);
  const uint32_t cw_ent = iter_word(a.iteration, kPurposeResidual);
  const bool vec_ok = ((((uintptr_t)tp) | ((uintptr_t)dp)) & 15) == 0;
  // block q of the lane set: groups 4 (set + q SETS) .. + 3 of the share
  uint4 qt[4 * Q], qd[4 * Q];
#pragma unroll
  for (int j = 0; j < 4 * Q; ++j) {
    const int gl = 4 * (set + j / 4 * SETS) + j % 4;
    qt[j] = gl < nloc ? load_logits<T>(tp, (gs + gl) * kGroup + sub * VEC, a.V, vec_ok) : neg_inf_vec<T>();
    qd[j] = bonus ? make_uint4(0, 0, 0, 0) : neg_inf_vec<T>();
    if (!bonus && gl < nloc) qd[j] = load_logits<T>(dp, (gs + gl) * kGroup + sub * VEC, a.V, vec_ok);
  }
  float e[Q];                            // the exponential of the lane's group of each block
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    const U4 wd = philox4x32_10(U4{(uint32_t)(gs / 4 + set + q * SETS), (uint32_t)b, (uint32_t)pos, cw_grp}, k0, k1);
    const int k = sub & 3;
    e[q] = expo(k == 0 ? wd.x : k == 1 ? wd.y : k == 2 ? wd.z : wd.w);
  }
  if (tid == 0) {
    sh.best[0] = ~0ull;
    sh.am = 0ull;
  }
  RowStat st{ts.x, 1.0f / ts.y, ds.x, -1.0f / ds.y};
  if (bonus) {                           // p relative to the row's largest logit
    float m = -pos_inf();
#pragma unroll
    for (int j = 0; j < 4 * Q; ++j) m = fmaxf(m, vec_max(qt[j], (const T*)nullptr));
    m = warp_max(m);
    if (lane == 0) sh.wmax[warp] = m;
    __syncthreads();
#pragma unroll
    for (int k = 0; k < NT / 32; ++k) m = fmaxf(m, sh.wmax[k]);
    if (tid < nc) *cl.map_shared_rank(&sh.ref[cr], tid) = m;
    cluster_sync();
    for (int c = 0; c < nc; ++c) m = fmaxf(m, sh.ref[c]);
    st = RowStat{mlog2e(m), 1.0f, 0.f, 0.f};
  } else {
    __syncthreads();
  }
  float key = pos_inf();
  int grp = kIntMax;
  const bool up1 = (sub & 1) != 0, up2 = (sub & 2) != 0;
#pragma unroll
  for (int q = 0; q < Q; ++q) {
    float s[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) s[k] = resid_vec<T>(qt[4 * q + k], qd[4 * q + k], st);
    const float x0 = (up1 ? s[1] : s[0]) + __shfl_xor_sync(kFull, up1 ? s[0] : s[1], 1);   // group 0 or 1
    const float x1 = (up1 ? s[3] : s[2]) + __shfl_xor_sync(kFull, up1 ? s[2] : s[3], 1);   // group 2 or 3
    float acc = (up2 ? x1 : x0) + __shfl_xor_sync(kFull, up2 ? x0 : x1, 2);
    if (LPG == 8) acc += __shfl_xor_sync(kFull, acc, 4);
    const int gl = 4 * (set + q * SETS) + (sub & 3);
    const float kq = (gl < nloc && acc > 0.f) ? e[q] / acc : pos_inf();
    if (kq < key) {                      // (a later block's groups are higher: ties keep the lower)
      key = kq;
      grp = gs + gl;
    }
  }
  // the CTA's least (key, group); the warp that holds that group races its
  // entries and pushes the result to rank 0 of the cluster
  key_min_cta(key, grp, &sh.best[0]);
  const int gw = grp != kIntMax ? grp - gs : 0;
  const int hs = gw / 4 % SETS;          // the lane set that holds it
  if (warp == hs * LPG / 32) {
    int tok = -1;
    if (grp != kIntMax) {
      const int j = gw / 4 / SETS * 4 + gw % 4;
      uint4 vt = qt[0], vd = qd[0];
#pragma unroll
      for (int k = 1; k < 4 * Q; ++k)
        if (j == k) {
          vt = qt[k];
          vd = qd[k];
        }
      tok = race_group_entries<T>(vt, vd, grp, hs * LPG % 32, lane, st, (uint32_t)b, (uint32_t)pos, cw_ent, k0, k1);
    }
    if (lane == 0) {
      *cl.map_shared_rank(&sh.rk[cr], 0) = key;
      *cl.map_shared_rank(&sh.rg[cr], 0) = grp;
      *cl.map_shared_rank(&sh.rt[cr], 0) = tok;
    }
  }
  cluster_sync();                        // every CTA's result is in rank 0
  if (cr == 0) draw_result<T, NT>(a, nc, b, pos, tp, vec_ok, sh);
}

template <typename T, int NT, int MODE, bool SAMPLED, bool SECOND>
__global__ void __launch_bounds__(NT, 512 / NT) seq_kernel(const StreamArgs a, const __grid_constant__ SeqSplit sp) {
  constexpr int NW = NT / 32;
  constexpr bool HAS_D = MODE != kModeVerify;
  constexpr bool HAS_T = MODE != kModeConf;
  constexpr int VEC = Elem<T>::kVec;
  extern __shared__ __align__(128) unsigned char seq_smem[];
  __shared__ SeqRow s_row[kSeqMaxK];
  // A tail's logits while its piece's vectors are reduced: in shared memory
  // where the loop has no two registers to spare (PAPER, in registers: spills,
  // and B=32 K=8 V=128256 26.4 us against 25.5), else in registers (the
  // drafter alone, in shared memory: spills, and B=64 K=1 V=50257 5.3 us
  // against 4.8).  The bf16 target alone, PAPER, requests them afterwards (B=48
  // K=8 V=64127 11.9 us; in registers 12.6, in shared memory 12.7).
  constexpr bool kStash = MODE == kModeFused;
  constexpr bool kLate = MODE == kModeVerify && !SAMPLED && VEC == 8;
  __shared__ float2 s_tail[kStash ? NW : 1][VEC - 1];
  cg::cluster_group cl = cg::this_cluster();
  const int nc = sp.nc;
  const int cr = (int)cl.block_rank(), b = (int)(blockIdx.x / (unsigned)nc);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nw = nc * NW;
  Partial* s_part = reinterpret_cast<Partial*>(seq_smem);
  // the warp's first piece: pieces are dealt over the CTAs in turn
  int kb = a.K, p = sp.pieces[kb], u = warp * nc + cr;
  SeqPiece<T> pc = {};
  if (!a.k_row) pc = seq_piece<T, MODE>(a, sp, b, u, p, sp.len[kb]);
  // A programmatic dependent of whatever precedes it on the stream: its CTAs
  // may be placed early, and wait here for that grid's completion.
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
  cluster_arrive();                      // (a peer's shared memory is written only after the matching wait)
  if (a.k_row) {
    const int raw = __ldg(a.k_row + b);
    kb = raw < 0 ? 0 : (raw > a.K ? a.K : raw);
    if (raw != kb && cr == 0 && threadIdx.x == 0) atomicOr(a.ws.err, 2u);
    p = sp.pieces[kb];
    if (kb > 0) pc = seq_piece<T, MODE>(a, sp, b, u, p, sp.len[kb]);
  }
  const int beta = a.beta_rank > 0 ? a.beta_rank : 0;
  // The window's drafted tokens, position i in lane i, and what the row merges
  // of this warp need, row warp + NW l in lane l: requested
  // here, used only once the slice's first logits are on their way.
  int tok = -1, tok_in = 0;
  if (HAS_T && lane < kb) tok = __ldg(a.tokens + (size_t)b * a.K + lane);
  float m_c = 0.f, m_zd = 0.f, m_lse = 0.f, m_conf = 0.f;
  auto row_inputs = [&]() {
    if (!HAS_T) return;
    if (lane < kb) {
      tok_in = tok;
      if (tok < 0 || tok >= a.V) {       // out-of-range draft: clamped, reported
        if (cr == 0 && warp == 0) atomicOr(a.ws.err, 1u);
        tok_in = 0;
      }
    }
    const int im = warp + NW * lane;
    const int tk = __shfl_sync(kFull, tok_in, im & 31);
    if (im < kb) {
      m_c = Elem<T>::load((const T*)a.target + ((size_t)b * a.Kt + im) * (size_t)a.V + tk);
      if (SAMPLED) m_zd = Elem<T>::load((const T*)a.draft + ((size_t)b * a.K + im) * (size_t)a.V + tk);
      if (MODE == kModeVerify) {
        m_conf = __ldg(a.conf_in + b * a.K + im);
        if (SAMPLED) m_lse = __ldg(a.lse_in + b * a.K + im);
      }
    }
  };
  bool first = true;                     // the warp has not reduced a segment yet
  while (u < kb * p) {
    const int i = pc.i, k = pc.k;
    const T* dp = pc.dp;
    const T* tp = pc.tp;
    const Seg sg = pc.sg;
    Pipe<T, HAS_D && HAS_T ? (SAMPLED ? CMSD_SEQ_UNROLL_S : CMSD_SEQ_UNROLL) : CMSD_SEQ_UNROLL1> pp;
    pipe_start<T, MODE>(pp, dp, tp, sg.va, sg.vb, lane);
    SegState ss;
    ss.c = ss.zd = 0.f;
    if (first) row_inputs();
    if (HAS_T) {
      const int tk = __shfl_sync(kFull, tok_in, i);
      ss.c = Elem<T>::load(tp + tk);
    }
    dlane_init(ss.d);
    tlane_init(ss.t, ss.c, beta);
    // The unaligned head (in the first lanes) and tail (in the last): requested
    // together, the head folded before the vectors and the tail after them, in
    // the order of a lane's indices (a vector takes the maximum's place on a
    // strict increase alone).
    const int hd = sg.va - sg.v0, tl = sg.v1 - sg.vb;
    const int ve = lane < hd ? sg.v0 + lane : sg.v1 - 32 + lane;
    float ze_d = 0.f, ze_t = 0.f;
    if (lane < hd || (!kLate && lane >= 32 - tl)) {
      if (HAS_D) ze_d = Elem<T>::load(dp + ve);
      if (HAS_T) ze_t = Elem<T>::load(tp + ve);
    }
    if (lane < hd) {
      if (HAS_D) d_scalar(ss.d, ze_d, ve);
      if (HAS_T) t_scalar<SAMPLED>(ss.t, ze_t, ve, ss.c, beta);
    } else if (kStash && lane >= 32 - tl) {
      s_tail[warp][lane - 33 + VEC] = make_float2(ze_d, ze_t);
    }
    pipe_run<T, MODE, SAMPLED>(pp, ss, sg.va, beta, lane);
    if (lane >= 32 - (sg.v1 - sg.vb)) {
      const int v = sg.v1 - 32 + lane;
      float2 z = make_float2(ze_d, ze_t);
      if (kStash) z = s_tail[warp][lane - 33 + VEC];
      if (kLate) z.y = Elem<T>::load(tp + v);
      if (HAS_D) d_scalar(ss.d, z.x, v);
      if (HAS_T) t_scalar<SAMPLED>(ss.t, z.y, v, ss.c, beta);
    }
    DRed dr;
    TRed tr;
    seg_reduce<T, MODE, SAMPLED>(ss, sg, !SAMPLED || a.argmax != nullptr, dp, tp, dr, tr);
    if (first) cluster_wait();         // every CTA of the cluster has started
    first = false;
    if (lane < nc) {                     // the partial into every CTA
      Partial q;
      q.d_m = dr.m; q.d_s = dr.s; q.d_t2 = dr.t2; q.d_top2 = dr.top2; q.d_idx = dr.idx;
      q.t_m = tr.m; q.t_s = tr.s; q.t_idx = tr.idx; q.t_cnt = tr.cnt;
      q.pad[0] = q.pad[1] = q.pad[2] = 0;
      *cl.map_shared_rank(s_part + i * p + k, lane) = q;
    }
    u += nw;
    if (u < kb * p) pc = seq_piece<T, MODE>(a, sp, b, u, p, sp.len[kb]);
  }
  if (first) {
    row_inputs();
    cluster_wait();
  }
  cluster_sync();                        // every CTA has every piece's partial
  // -- rows: every CTA merges and decides all of them (a second exchange and
  // barrier took longer), CTA 0 writes their outputs -----------------------------
  for (int l = 0, i = warp; i < kb; i += NW, ++l) {
    DRed dm = dred_empty();
    TRed tm = tred_empty();
    for (int k = lane; k < p; k += 32) {
      const float4* src = reinterpret_cast<const float4*>(s_part + i * p + k);
      const float4 x0 = src[0], x1 = src[1], x2 = src[2];
      if (HAS_D) fold_d(dm, DRed{x0.x, x0.y, x0.z, x0.w, __float_as_int(x1.x)});
      if (HAS_T) fold_t(tm, TRed{x1.y, x1.z, __float_as_int(x1.w), __float_as_int(x2.x)});
    }
    const DRed dr = HAS_D ? reduce_d(dm) : dred_empty();
    const TRed tr = HAS_T ? reduce_t(tm) : tred_empty();
    const RowOut o = row_results<MODE, SAMPLED>(a, b * a.K + i, b, i, dr, tr, __shfl_sync(kFull, m_c, l),
                                                __shfl_sync(kFull, m_zd, l), __shfl_sync(kFull, m_lse, l),
                                                __shfl_sync(kFull, m_conf, l), lane, cr == 0);
    if (lane == 0) {
      SeqRow q;
      q.stat = make_float4(o.ds.x, o.ds.y, o.ts.x, o.ts.y);
      q.cfx = o.cfx;
      q.acc = o.acc ? 1 : 0;
      q.pad = 0;
      s_row[i] = q;
    }
  }
  __syncthreads();
  // -- the sequence ---------------------------------------------------------------
  const bool have = lane < kb;
  const bool acc = have && s_row[lane & (kSeqMaxK - 1)].acc != 0;
  const unsigned rej = __ballot_sync(kFull, have && !acc);
  const int n = (HAS_T && rej) ? __ffs(rej) - 1 : kb;
  if (cr == 0 && warp == 0) {
    if (HAS_D && a.k_next) {
      unsigned long long cs = have ? s_row[lane & (kSeqMaxK - 1)].cfx : 0ull;
#pragma unroll
      for (int o = 16; o; o >>= 1) cs += __shfl_xor_sync(kFull, cs, o);
      if (lane == 0) a.k_next[b] = next_k(a, cs, kb);
    }
    if (HAS_T) {
      if (lane == 0) a.n_accept[b] = n;
      write_outputs<MODE, SAMPLED>(a, b, kb, n, lane, tok, acc);
    }
  }
  if (SECOND) {
    const int kind = seq_kind<MODE, SAMPLED>(a, n, kb);      // the same in every thread of the cluster
    if (kind == kSeqNone) return;
    // the draw's state follows the partials, which a peer may still be merging
    unsigned char* draw = seq_smem + sp.part_bytes;
    DrawShared<T, NT>& sh = *reinterpret_cast<DrawShared<T, NT>*>(draw);
    float* s_u = reinterpret_cast<float*>(draw + sizeof(DrawShared<T, NT>));
    const T* tp = (const T*)a.target + ((size_t)b * a.Kt + n) * (size_t)a.V;
    if (!SAMPLED) {
      cluster_argmax<T, NT>(a, cl, nc, cr, b, n, tp, sh);
      return;
    }
    const bool bonus = kind == kSeqBonus;
    const float4 q = bonus ? make_float4(0.f, 1.f, 0.f, 1.f) : s_row[n].stat;
    const T* dp = bonus ? tp : (const T*)a.draft + ((size_t)b * a.K + n) * (size_t)a.V;
    const float2 ts = make_float2(q.z, q.w), ds = make_float2(q.x, q.y);
    const int ngs = draw_share((a.V + kGroup - 1) / kGroup, nc);
    const bool aligned = ((((uintptr_t)tp) | ((uintptr_t)dp)) & 15) == 0;
    if (ngs <= 4 * DrawShared<T, NT>::kSets)
      cluster_race<T, NT, 1>(a, cl, nc, cr, b, n, bonus, tp, dp, ts, ds, sh);
    else if (aligned && ngs <= 8 * DrawShared<T, NT>::kSets)
      cluster_race<T, NT, 2>(a, cl, nc, cr, b, n, bonus, tp, dp, ts, ds, sh);
    else
      cluster_draw<T, NT, 4>(a, cl, nc, cr, b, n, bonus, tp, dp, ts, ds, s_u, sh);
  }
}

// How the rows of a window of kb positions are cut: `pieces` near-equal
// pieces of `len` entries (a multiple of a 128-byte line) each, dealt to the
// cluster's nw warps in turn.  Every m-th multiple of the warps is tried: more
// pieces balance better, and each piece costs its warp a reduction, about the
// time of two stages of loads.  At most 64 pieces per row (two partials per
// lane in the row merge).
template <typename T>
void seq_split_window(SeqSplit& sp, int kb, int V, int nw) {
  const int line = 128 / (int)sizeof(T);
  const int cost = 2 * CMSD_SEQ_UNROLL * 32 * Elem<T>::kVec;
  long long best = 0;
  sp.pieces[kb] = 1;
  sp.len[kb] = V;
  for (int m = 1; m <= 4; ++m) {
    int p = m * nw / kb;
    p = p < 1 ? 1 : (p > 64 ? 64 : p);
    int len = (V + p - 1) / p;
    if (len < 2 * 32 * Elem<T>::kVec) len = 2 * 32 * Elem<T>::kVec;   // two vectors per lane
    len = (len + line - 1) / line * line;
    p = (V + len - 1) / len;
    const long long t = (long long)((kb * p + nw - 1) / nw) * (len + cost);
    if (m == 1 || t < best) {
      best = t;
      sp.pieces[kb] = (short)p;
      sp.len[kb] = len;
    }
  }
}

// The window's partials, then the draw's state and its share's uniforms and
// bounds.
template <typename T, int NT>
size_t seq_smem_bytes(SeqSplit& sp, int k0, int K, int V, bool second, bool sampled) {
  int slots = 0;
  for (int k = k0; k <= K; ++k) {
    const int n = k * sp.pieces[k];
    slots = n > slots ? n : slots;
  }
  sp.part_bytes = (int)((slots * sizeof(Partial) + 127) / 128 * 128);
  return (size_t)sp.part_bytes + (second ? sizeof(DrawShared<T, NT>) + (sampled ? draw_smem_bytes(V, sp.nc) : 0) : 0);
}
// (two CTAs of 256 threads, or one of 512, fit an SM with this much each)
constexpr size_t kSeqSmemMax = 112 * 1024;

template <typename T, int NT, int MODE, bool SAMPLED, bool SECOND>
cudaError_t seq_attrs() {
  static unsigned long long done = 0ull;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const unsigned long long bit = 1ull << (dev & 63);
  if (__atomic_load_n(&done, __ATOMIC_ACQUIRE) & bit) return cudaSuccess;
  auto kernel = seq_kernel<T, NT, MODE, SAMPLED, SECOND>;
  e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSeqSmemMax);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e == cudaSuccess) __atomic_fetch_or(&done, bit, __ATOMIC_ACQ_REL);
  return e;
}

inline void seq_config(cudaLaunchConfig_t& cfg, cudaLaunchAttribute (&attr)[2], int B, int nc, int threads, size_t smem) {
  cfg = {};
  cfg.gridDim = dim3((unsigned)(B * nc));
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)nc;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
}

// Clusters of nc CTAs that can be resident on the current device, for the
// variant with the most registers and any row's shared memory (0: none).
template <typename T, int NT>
int seq_clusters_t(int nc) {
  if (seq_attrs<T, NT, kModeFused, true, true>() != cudaSuccess) return 0;
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr[2];
  seq_config(cfg, attr, 1, nc, NT, kSeqSmemMax);
  cfg.numAttrs = 1;                      // the cluster size
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, seq_kernel<T, NT, kModeFused, true, true>, &cfg) != cudaSuccess) {
    (void)cudaGetLastError();            // a refused query leaves no error behind for the caller
    return 0;
  }
  return n;
}

template <typename T, int NT, int MODE, bool SAMPLED, bool SECOND>
cudaError_t launch_seq_one(const StreamArgs& a, int nc, cudaStream_t s) {
  const cudaError_t e = seq_attrs<T, NT, MODE, SAMPLED, SECOND>();
  if (e != cudaSuccess) return e;
  SeqSplit sp = {};
  sp.nc = nc;
  const int k0 = a.k_row ? 1 : a.K;
  for (int k = k0; k <= a.K; ++k) seq_split_window<T>(sp, k, a.V, nc * (NT / 32));
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr[2];
  seq_config(cfg, attr, a.B, nc, NT, seq_smem_bytes<T, NT>(sp, k0, a.K, a.V, SECOND, SAMPLED));
  cfg.stream = s;
  return cudaLaunchKernelEx(&cfg, seq_kernel<T, NT, MODE, SAMPLED, SECOND>, a, sp);
}

template <typename T, int NT>
cudaError_t launch_seq_t(int mode, bool sampled, bool second, const StreamArgs& a, int nc, cudaStream_t s) {
  if (mode == kModeConf) return launch_seq_one<T, NT, kModeConf, false, false>(a, nc, s);
  if (mode == kModeVerify) {
    if (sampled) return launch_seq_one<T, NT, kModeVerify, true, true>(a, nc, s);
    if (second) return launch_seq_one<T, NT, kModeVerify, false, true>(a, nc, s);
    return launch_seq_one<T, NT, kModeVerify, false, false>(a, nc, s);
  }
  if (sampled) return launch_seq_one<T, NT, kModeFused, true, true>(a, nc, s);
  if (second) return launch_seq_one<T, NT, kModeFused, false, true>(a, nc, s);
  return launch_seq_one<T, NT, kModeFused, false, false>(a, nc, s);
}

// Whether the state of a draw over rows of V entries fits, whatever the
// cluster's size.
template <typename T>
bool seq_draw_fits_t(int V) {
  const size_t parts = 4 * kSeqMaxCtas * 16 * sizeof(Partial);   // four pieces per warp, CTAs of 512 threads
  return parts + sizeof(DrawShared<T, 512>) + draw_smem_bytes(V, 1) <= kSeqSmemMax;
}

}  // namespace cmsd
