// The logits pass in one launch, a thread-block cluster per sequence (sm_103a).
//
// For windows of at most 16 positions and problems too small to fill the
// streaming kernel's grid for long (the rule is seq_cluster in cmsd_api.cu).
// There the time is not bandwidth but the chain of dependent steps, and the
// streaming kernel's chain goes through global memory: partials and an
// acquire-release atomic per slice, loads of them by the row's merger, an
// atomic per row, a record word and a second kernel that polls it, each step
// an L2 round trip of about a microsecond.  Here a sequence's rows are cut
// over the warps of one cluster and every hand-over is a store into a peer's
// shared memory and a cluster barrier:
//   stream   each warp reduces its slice (the streaming kernel's arithmetic,
//            four vectors per tensor and lane in flight ahead of the four
//            being reduced) and stores its partial into the CTA that merges
//            the row (row i: CTA i mod nc);
//   rows     barrier; one warp per row merges its partials, takes the row's
//            decision and stores it into every CTA;
//   sequence barrier; every CTA finds the first rejection, CTA 0 writes the
//            sequence's outputs;
//   draw     under the sampled rule, or for the bonus row, the cluster draws
//            the token itself: the race by group bounds (cluster_draw).
#pragma once
#include "cmsd_stream_impl.cuh"

namespace cmsd {

constexpr int kSeqMaxCtas = 16;          // CTAs per cluster (16: a non-portable size)
constexpr int kSeqMaxK = kPackedMaxK;    // positions per window
#ifndef CMSD_SEQ_UNROLL
#define CMSD_SEQ_UNROLL 4
#endif
#ifndef CMSD_SEQ_UNROLL1
#define CMSD_SEQ_UNROLL1 8
#endif
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }
__device__ __forceinline__ void cluster_sync() {
  cluster_arrive();
  cluster_wait();
}

// ---------------------------------------------------------------------------
// the draw by group bounds, by the cluster that holds the sequence
// ---------------------------------------------------------------------------
//
// The race of resample_bound_kernel (bound, probe, race, level 2; the same
// keys, filter and tie rule), with the group maxima taken from global memory:
// the row was streamed moments ago and comes from L2, so it is not staged.
// The bonus race is the same with r = p, p relative to the row's maximum
// (the normaliser does not change the order of the keys).

constexpr int kDrawCands = 1024;         // candidate list; past it the share is raced whole

template <typename T, int NT>
struct DrawShared {
  static constexpr int kLpg = kGroup / Elem<T>::kVec;     // lanes per group
  static constexpr int kSets = NT / kLpg;                 // lane sets per CTA
  unsigned long long best[2];            // key_min_cta of the probes, of the race
  unsigned long long am;                 // rank 0: row_argmax_cta's reduction
  unsigned long long arg[kSeqMaxCtas];   // rank 0: each CTA's (value, ~index) of the bonus argmax
  uint4 qt[NT], qd[NT];                  // vectors of each lane set's best group
  int probe[kSets];                      // the group each lane set probed
  int list[kDrawCands];
  float ref[kSeqMaxCtas];                // each CTA's largest logit (bonus race)
  float k1[kSeqMaxCtas];                 // each CTA's least probe key
  float rk[kSeqMaxCtas];                 // rank 0: each CTA's (key, group, token)
  int rg[kSeqMaxCtas], rt[kSeqMaxCtas];
  float wmax[NT / 32];
  int n, hold, fb;
};

// Groups per CTA of an nc-CTA cluster: a multiple of four, so that a share
// starts on a block of four group uniforms.
__host__ __device__ inline int draw_share(int ng, int nc) { return ((ng + nc - 1) / nc + 3) & ~3; }
// dynamic shared memory of the draw: the share's uniforms and bounds
__host__ __device__ inline size_t draw_smem_bytes(int V, int nc) {
  return (size_t)draw_share((V + kGroup - 1) / kGroup, nc) * 2 * sizeof(float);
}

template <typename T, int NT>
__device__ void cluster_draw(const StreamArgs& a, cg::cluster_group& cl, int nc, int cr, int b, int pos, bool bonus,
                             const T* tp, const T* dp, RowStat st, float* s_u, DrawShared<T, NT>& sh) {
  constexpr int VEC = Elem<T>::kVec;
  constexpr int LPG = DrawShared<T, NT>::kLpg;
  constexpr int SETS = DrawShared<T, NT>::kSets;
  constexpr int UL = 4;                  // vectors in flight per thread of the maxima pass
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int sub = lane % LPG, set = tid / LPG;
  const int ng = (a.V + kGroup - 1) / kGroup;
  const int ngs = draw_share(ng, nc);
  const int gs = cr * ngs;                                   // the share: groups [gs, gs + nloc)
  const int nloc = max(0, min(ng, gs + ngs) - gs);
  float* s_rb = s_u + ngs;
  const uint32_t k0 = seed_lo(a.seed), k1 = seed_hi(a.seed);
  const uint32_t cw_grp = iter_word(a.iteration, kPurposeGroup);
  const uint32_t cw_ent = iter_word(a.iteration, kPurposeResidual);
  const bool vec_ok = ((((uintptr_t)tp) | ((uintptr_t)dp)) & 15) == 0;
  if (tid == 0) {
    sh.best[0] = sh.best[1] = ~0ull;
    sh.am = 0ull;
    sh.n = 0;
    sh.hold = 0;
  }
  // largest logit of each group of the share (-inf past the row end)
  const int nv = nloc * LPG, v0 = gs * kGroup;
  for (int j0 = 0; j0 < nv; j0 += NT * UL) {
    uint4 q[UL];
#pragma unroll
    for (int k = 0; k < UL; ++k) {
      const int j = j0 + k * NT + tid;
      q[k] = j < nv ? load_logits<T>(tp, v0 + j * VEC, a.V, vec_ok) : neg_inf_vec<T>();
    }
#pragma unroll
    for (int k = 0; k < UL; ++k) {
      const int j = j0 + k * NT + tid;
      float m = vec_max(q[k], (const T*)nullptr);
#pragma unroll
      for (int o = 1; o < LPG; o <<= 1) m = fmaxf(m, __shfl_xor_sync(kFull, m, o));
      if (sub == 0 && j < nv) s_rb[j / LPG] = m;
    }
  }
  for (int q = tid; q < (nloc + 3) / 4; q += NT) {
    const U4 wd = philox4x32_10(U4{(uint32_t)(gs / 4 + q), (uint32_t)b, (uint32_t)pos, cw_grp}, k0, k1);
    s_u[4 * q + 0] = word_to_unit(wd.x);
    s_u[4 * q + 1] = word_to_unit(wd.y);
    s_u[4 * q + 2] = word_to_unit(wd.z);
    s_u[4 * q + 3] = word_to_unit(wd.w);
  }
  __syncthreads();
  if (bonus) {                           // p relative to the row's largest logit
    float m = -pos_inf();
    for (int gl = tid; gl < nloc; gl += NT) m = fmaxf(m, s_rb[gl]);
    m = warp_max(m);
    if (lane == 0) sh.wmax[warp] = m;
    __syncthreads();
#pragma unroll
    for (int k = 0; k < NT / 32; ++k) m = fmaxf(m, sh.wmax[k]);
    if (tid < nc) *cl.map_shared_rank(&sh.ref[cr], tid) = m;
    cluster_sync();
    for (int c = 0; c < nc; ++c) m = fmaxf(m, sh.ref[c]);
    st = RowStat{mlog2e(m), 1.0f, 0.f, 0.f};
  }
  // bound: each thread keeps its lowest U_g / Rb_g (compared as U_a Rb_b <
  // U_b Rb_a), then each lane set the lowest of its LPG threads'
  float bu = 0.f, brb = 1.f;
  int lg = -1;
  for (int gl = tid; gl < nloc; gl += NT) {
    const float rb = group_bound(s_rb[gl], st);
    s_rb[gl] = rb;
    const float u = s_u[gl];
    if (lg < 0 || u * brb < bu * rb) {
      bu = u;
      brb = rb;
      lg = gl;
    }
  }
#pragma unroll
  for (int o = 1; o < LPG; o <<= 1) {
    const float u2 = __shfl_xor_sync(kFull, bu, o), rb2 = __shfl_xor_sync(kFull, brb, o);
    const int g2 = __shfl_xor_sync(kFull, lg, o);
    if (g2 >= 0 && (lg < 0 || u2 * brb < bu * rb2 || (u2 * brb == bu * rb2 && g2 < lg))) {
      bu = u2;
      brb = rb2;
      lg = g2;
    }
  }
  // probe: the lane set's lowest-bound group, exactly
  float sk = pos_inf();                  // the lane set's best (key, group), its vectors in qt, qd
  int sg = kIntMax;
  {
    uint4 qt = neg_inf_vec<T>(), qd = bonus ? make_uint4(0, 0, 0, 0) : neg_inf_vec<T>();
    if (lg >= 0) {
      qt = load_logits<T>(tp, (gs + lg) * kGroup + sub * VEC, a.V, vec_ok);
      if (!bonus) qd = load_logits<T>(dp, (gs + lg) * kGroup + sub * VEC, a.V, vec_ok);
    }
    sk = group_key<T>(qt, qd, st, lg >= 0 ? s_u[lg] : 0.f, lg >= 0);
    sg = sk != pos_inf() ? gs + lg : kIntMax;
    sh.qt[tid] = qt;
    sh.qd[tid] = qd;
    if (sub == 0) sh.probe[set] = lg;
  }
  float K1 = sk;
  int g1 = sg;
  key_min_cta(K1, g1, &sh.best[0]);
  // K1: the least probe key of the cluster, an upper bound on the winner's key
  if (tid < nc) *cl.map_shared_rank(&sh.k1[cr], tid) = K1;
  cluster_sync();
  for (int c = 0; c < nc; ++c) K1 = fminf(K1, sh.k1[c]);
  // race: the groups of the share that the bound leaves at or below K1 and
  // that no lane set has probed
  for (int gl = tid; gl < nloc; gl += NT) {
    if (!(s_u[gl] * kRaceFilter > K1 * s_rb[gl]) && sh.probe[(gl % NT) / LPG] != gl) {
      const int i = atomicAdd(&sh.n, 1);
      if (i < kDrawCands) sh.list[i] = gl;
    }
  }
  __syncthreads();
  const int ncand = sh.n;
  const bool whole = ncand > kDrawCands;
  const int items = whole ? nloc : ncand;
  for (int i0 = 0; i0 < items; i0 += SETS) {                 // block-uniform trip count
    const int i = i0 + set;
    const int gl = i < items ? (whole ? i : sh.list[i]) : -1;
    uint4 qt = neg_inf_vec<T>(), qd = bonus ? make_uint4(0, 0, 0, 0) : neg_inf_vec<T>();
    if (gl >= 0) {
      qt = load_logits<T>(tp, (gs + gl) * kGroup + sub * VEC, a.V, vec_ok);
      if (!bonus) qd = load_logits<T>(dp, (gs + gl) * kGroup + sub * VEC, a.V, vec_ok);
    }
    const float key = group_key<T>(qt, qd, st, gl >= 0 ? s_u[gl] : 0.f, gl >= 0);
    if (key != pos_inf() && (key < sk || (key == sk && gs + gl < sg))) {   // the whole lane set agrees
      sk = key;
      sg = gs + gl;
      sh.qt[tid] = qt;
      sh.qd[tid] = qd;
    }
  }
  // the CTA's least (key, group), the lane set holding it, and its level-2
  // winner, pushed to rank 0 of the cluster
  float ck = sk;
  int cgrp = sg;
  key_min_cta(ck, cgrp, &sh.best[1]);
  if (sub == 0 && cgrp != kIntMax && sk == ck && sg == cgrp) sh.hold = set;   // holders share one group
  __syncthreads();
  if (warp == 0) {
    int tok = -1;
    if (cgrp != kIntMax) {
      const int h = sh.hold;
      tok = race_group_entries<T>(sh.qt[h * LPG + sub], sh.qd[h * LPG + sub], cgrp, 0, lane, st, (uint32_t)b,
                                  (uint32_t)pos, cw_ent, k0, k1);
    }
    if (lane == 0) {
      *cl.map_shared_rank(&sh.rk[cr], 0) = ck;
      *cl.map_shared_rank(&sh.rg[cr], 0) = cgrp;
      *cl.map_shared_rank(&sh.rt[cr], 0) = tok;
    }
  }
  cluster_sync();                             // every CTA's result is in rank 0
  if (cr == 0) {
    if (warp == 0) {
      float k = lane < nc ? sh.rk[lane] : pos_inf();
      const int g = lane < nc ? sh.rg[lane] : kIntMax;
      const uint32_t kb = __reduce_min_sync(kFull, __float_as_uint(k));      // keys are >= 0 or +inf
      const uint32_t gb = __reduce_min_sync(kFull, __float_as_uint(k) == kb ? (uint32_t)g : 0xFFFFFFFFu);
      const unsigned who = __ballot_sync(kFull, __float_as_uint(k) == kb && (uint32_t)g == gb);
      const int c = __ffs(who) - 1;
      if (lane == 0) sh.fb = (gb == (uint32_t)kIntMax || sh.rt[c] < 0) ? -1 : sh.rt[c];
    }
    __syncthreads();
    int tok = sh.fb;
    if (tok < 0) tok = row_argmax_cta<T, NT>(tp, a.V, vec_ok, &sh.am);   // empty residual: the argmax
    if (tid == 0) a.out_tokens[(size_t)b * a.Ko + pos] = tok;
  }
}

// The extra verifier row's argmax (PAPER rule, bonus row; lowest index), each
// CTA a share of the row.
template <typename T, int NT>
__device__ void cluster_argmax(const StreamArgs& a, cg::cluster_group& cl, int nc, int cr, int b, int pos, const T* tp,
                               DrawShared<T, NT>& sh) {
  constexpr int VEC = Elem<T>::kVec;
  const int tid = threadIdx.x;
  const bool vec_ok = (((uintptr_t)tp) & 15) == 0;
  const int nvec = (a.V + VEC - 1) / VEC;
  const int per = (nvec + nc - 1) / nc;
  const int j1 = min(nvec, (cr + 1) * per);
  if (tid == 0) sh.am = 0ull;
  float bm = -pos_inf();
  int bi = kIntMax;
  for (int j = cr * per + tid; j < j1; j += NT) {
    const uint4 q = load_logits<T>(tp, j * VEC, a.V, vec_ok);
#pragma unroll
    for (int k = 0; k < VEC; ++k) {
      const float z = logit_at<T>(q, k);
      if (j * VEC + k < a.V && (z > bm || (z == bm && j * VEC + k < bi))) {
        bm = z;
        bi = j * VEC + k;
      }
    }
  }
  __syncthreads();
  const unsigned long long key = argmax_key_cta(bm, bi, &sh.am);
  if (tid == 0) *cl.map_shared_rank(&sh.arg[cr], 0) = key;
  cluster_sync();
  if (cr == 0 && tid == 0) {
    unsigned long long m = 0ull;
    for (int c = 0; c < nc; ++c) m = max(m, sh.arg[c]);
    a.out_tokens[(size_t)b * a.Ko + pos] = (int)~(uint32_t)m;
  }
}

// ---------------------------------------------------------------------------
// the kernel
// ---------------------------------------------------------------------------

// The cut of a window of kb rows over the cluster's warps, by kb.
struct SeqSplit {
  int nc;                                // CTAs per cluster
  int rcp;                               // 65536 / nc + 1: i / nc = i rcp >> 16 for i <= kSeqMaxK
  int len[kSeqMaxK + 1];                 // entries per piece
  short pieces[kSeqMaxK + 1];            // pieces per row
};

// A row's decision as every CTA of the cluster keeps it.
struct __align__(16) SeqRow {
  float4 stat;                           // sampled rule: drafter, then target (max * log2e, sum)
  unsigned long long cfx;
  int acc, pad;
};

template <typename T, int NT, int MODE, bool SAMPLED, bool SECOND>
__global__ void __launch_bounds__(NT, 512 / NT) seq_kernel(const StreamArgs a, const __grid_constant__ SeqSplit sp) {
  constexpr int NW = NT / 32;
  constexpr bool HAS_D = MODE != kModeVerify;
  constexpr bool HAS_T = MODE != kModeConf;
  constexpr int VEC = Elem<T>::kVec;
  extern __shared__ __align__(128) unsigned char seq_smem[];
  __shared__ SeqRow s_row[kSeqMaxK];
  cg::cluster_group cl = cg::this_cluster();
  // A programmatic dependent of whatever precedes it on the stream: its CTAs
  // may be placed early, and wait here for that grid's completion.
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
  cluster_arrive();                      // (a peer's shared memory is written only after the matching wait)
  const int nc = sp.nc;
  const int cr = (int)cl.block_rank(), b = (int)(blockIdx.x / (unsigned)nc);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int w = warp * nc + cr;          // pieces are dealt over the CTAs in turn
  const int nw = nc * NW;
  Partial* s_part = reinterpret_cast<Partial*>(seq_smem);
  int kb = a.K;
  if (a.k_row) {
    const int raw = __ldg(a.k_row + b);
    kb = raw < 0 ? 0 : (raw > a.K ? a.K : raw);
    if (raw != kb && cr == 0 && threadIdx.x == 0) atomicOr(a.ws.err, 2u);
  }
  const int beta = a.beta_rank > 0 ? a.beta_rank : 0;
  // The window's drafted tokens, position i in lane i, and what the row merges
  // of this warp need, row cr + nc (warp + NW l) in lane l: requested
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
    const int im = cr + nc * (warp + NW * lane);
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
  const int p = sp.pieces[kb], len = sp.len[kb];
  for (int u = w; u < kb * p; u += nw) {
    const int i = (int)((unsigned)u / (unsigned)p), k = u - i * p;
    const int ic = (i * sp.rcp) >> 16;   // i / nc
    const T* dp = (const T*)a.draft + ((size_t)b * a.K + i) * (size_t)a.V;
    const T* tp = HAS_T ? (const T*)a.target + ((size_t)b * a.Kt + i) * (size_t)a.V : nullptr;
    const Seg sg = seg_geom<T>(HAS_D ? dp : tp, k * len, a.V, len);
    Pipe<T, HAS_D && HAS_T ? CMSD_SEQ_UNROLL : CMSD_SEQ_UNROLL1> pp;
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
    // the unaligned head (in the first lanes) and tail (in the last); after the
    // pipeline instead, the sampled rule's stages compiled to slower code (36
    // against 33.5 us at B=32 K=8 V=128256 with the bonus row)
    const int hd = sg.va - sg.v0, tl = sg.v1 - sg.vb;
    if (lane < hd || lane >= 32 - tl) {
      const int v = lane < hd ? sg.v0 + lane : sg.v1 - 32 + lane;
      if (HAS_D) d_scalar(ss.d, Elem<T>::load(dp + v), v);
      if (HAS_T) t_scalar<SAMPLED>(ss.t, Elem<T>::load(tp + v), v, ss.c, beta);
    }
    pipe_run<T, MODE, SAMPLED>(pp, ss, sg.va, beta, lane);
    DRed dr;
    TRed tr;
    seg_reduce<T, MODE, SAMPLED>(ss, !SAMPLED || a.argmax != nullptr, !SAMPLED, dp, tp, dr, tr);
    if (first) cluster_wait();         // every CTA of the cluster has started
    first = false;
    if (lane == 0) {
      Partial q;
      q.d_m = dr.m; q.d_s = dr.s; q.d_t2 = dr.t2; q.d_top2 = dr.top2; q.d_idx = dr.idx;
      q.t_m = tr.m; q.t_s = tr.s; q.t_idx = tr.idx; q.t_cnt = tr.cnt;
      q.pad[0] = q.pad[1] = q.pad[2] = 0;
      *cl.map_shared_rank(s_part + ic * p + k, i - ic * nc) = q;
    }
  }
  if (first) {
    row_inputs();
    cluster_wait();
  }
  cluster_sync();                        // every slice's partial is in its row's CTA
  // -- rows: merge, decide, tell every CTA ---------------------------------------
  for (int l = 0, i = cr + nc * warp; i < kb; i += nw, ++l) {
    DRed dm = dred_empty();
    TRed tm = tred_empty();
    for (int k = lane; k < p; k += 32) {
      const float4* src = reinterpret_cast<const float4*>(s_part + ((i * sp.rcp) >> 16) * p + k);
      const float4 x0 = src[0], x1 = src[1], x2 = src[2];
      if (HAS_D) fold_d(dm, DRed{x0.x, x0.y, x0.z, x0.w, __float_as_int(x1.x)});
      if (HAS_T) fold_t(tm, TRed{x1.y, x1.z, __float_as_int(x1.w), __float_as_int(x2.x)});
    }
    const DRed dr = HAS_D ? reduce_d(dm) : dred_empty();
    const TRed tr = HAS_T ? reduce_t(tm) : tred_empty();
    const RowOut o = row_results<MODE, SAMPLED>(a, b * a.K + i, b, i, dr, tr, __shfl_sync(kFull, m_c, l),
                                                __shfl_sync(kFull, m_zd, l), __shfl_sync(kFull, m_lse, l),
                                                __shfl_sync(kFull, m_conf, l), lane);
    if (lane < nc) {
      SeqRow q;
      q.stat = make_float4(o.ds.x, o.ds.y, o.ts.x, o.ts.y);
      q.cfx = o.cfx;
      q.acc = o.acc ? 1 : 0;
      q.pad = 0;
      *cl.map_shared_rank(s_row + i, lane) = q;
    }
  }
  cluster_sync();                        // every CTA has every row's decision
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
    // the partials have been merged: the draw's state takes their place
    DrawShared<T, NT>& sh = *reinterpret_cast<DrawShared<T, NT>*>(seq_smem);
    float* s_u = reinterpret_cast<float*>(seq_smem + sizeof(DrawShared<T, NT>));
    const T* tp = (const T*)a.target + ((size_t)b * a.Kt + n) * (size_t)a.V;
    if (!SAMPLED) {
      cluster_argmax<T, NT>(a, cl, nc, cr, b, n, tp, sh);
      return;
    }
    const bool bonus = kind == kSeqBonus;
    RowStat st{0.f, 1.f, 0.f, 0.f};
    const T* dp = tp;
    if (!bonus) {
      const float4 q = s_row[n].stat;
      st = RowStat{q.z, 1.0f / q.w, q.x, -1.0f / q.y};
      dp = (const T*)a.draft + ((size_t)b * a.K + n) * (size_t)a.V;
    }
    cluster_draw<T, NT>(a, cl, nc, cr, b, n, bonus, tp, dp, st, s_u, sh);
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

// The partials of the rows a CTA merges; the draw's state and its share's
// uniforms and bounds take their place.
template <typename T, int NT>
size_t seq_smem_bytes(const SeqSplit& sp, int K, int V, bool second, bool sampled) {
  const int nc = sp.nc;
  int slots = 0;
  for (int k = 1; k <= K; ++k) {
    const int n = ((k + nc - 1) / nc) * sp.pieces[k];
    slots = n > slots ? n : slots;
  }
  const size_t p = (size_t)slots * sizeof(Partial);
  const size_t d = second ? sizeof(DrawShared<T, NT>) + (sampled ? draw_smem_bytes(V, nc) : 0) : 0;
  return p > d ? p : d;
}
// (two CTAs of 256 threads, or one of 512, fit an SM with this much each)
constexpr size_t kSeqSmemMax = 96 * 1024;

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
  sp.rcp = 65536 / nc + 1;
  for (int k = a.k_row ? 1 : a.K; k <= a.K; ++k) seq_split_window<T>(sp, k, a.V, nc * (NT / 32));
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr[2];
  seq_config(cfg, attr, a.B, nc, NT, seq_smem_bytes<T, NT>(sp, a.K, a.V, SECOND, SAMPLED));
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
  return sizeof(DrawShared<T, 512>) + draw_smem_bytes(V, 1) <= kSeqSmemMax;
}

}  // namespace cmsd
