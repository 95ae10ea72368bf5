// C ABI of libcmsd.so: argument checks, workspace layout, launches, timing.
// The operations are specified in include/cmsd.h.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include <string.h>

#include <atomic>
#include <map>
#include <mutex>
#include <tuple>
#include <vector>

#include "cmsd.h"
#include "cmsd_internal.h"
#include "cmsd_philox.cuh"

using namespace cmsd;

namespace {

thread_local int g_last_cuda = 0;

int cuda_fail(cudaError_t e) {
  g_last_cuda = (int)e;
  return CMSD_ECUDA;
}

std::mutex g_mu;
std::map<int, int> g_sms;                                   // device -> SM count
std::map<std::tuple<int, int, int, int, int>, int> g_occ;   // (dev, dtype, mode, variant, smem) -> blocks/SM
std::map<std::tuple<int, int, int, int>, int> g_draw_res;    // (dev, dtype, V, CTAs) -> resident clusters
std::map<std::tuple<int, int, int>, int> g_occ_res;          // (dev, dtype, sampled) -> blocks/SM

int device_sms(int* sms) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return cuda_fail(e);
  std::lock_guard<std::mutex> lk(g_mu);
  auto it = g_sms.find(dev);
  if (it == g_sms.end()) {
    int n = 0;
    e = cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return cuda_fail(e);
    it = g_sms.emplace(dev, n).first;
  }
  *sms = it->second;
  return CMSD_OK;
}

int stream_grid(int dtype, int mode, bool sampled, bool second, int threads, size_t smem, int* grid) {
  int sms = 0;
  int rc = device_sms(&sms);
  if (rc) return rc;
  int dev = 0;
  cudaGetDevice(&dev);
  const int variant = (sampled ? 1 : 0) | (second ? 2 : 0) | threads << 2;
  const auto key = std::make_tuple(dev, dtype, mode, variant, (int)smem);
  std::lock_guard<std::mutex> lk(g_mu);
  auto it = g_occ.find(key);
  if (it == g_occ.end()) {
    int nb = 0;
    cudaError_t e = occupancy_stream(dtype, mode, sampled, second, threads, smem, &nb);
    if (e != cudaSuccess) return cuda_fail(e);
    if (nb < 1) nb = 1;
    it = g_occ.emplace(key, nb).first;
  }
  *grid = sms * it->second;
  return CMSD_OK;
}

int resample_grid(int dtype, bool sampled, int* grid) {
  int sms = 0;
  int rc = device_sms(&sms);
  if (rc) return rc;
  int dev = 0;
  cudaGetDevice(&dev);
  const auto key = std::make_tuple(dev, dtype, sampled ? 1 : 0);
  std::lock_guard<std::mutex> lk(g_mu);
  auto it = g_occ_res.find(key);
  if (it == g_occ_res.end()) {
    int nb = 0;
    cudaError_t e = occupancy_resample(dtype, sampled, &nb);
    if (e != cudaSuccess) return cuda_fail(e);
    if (nb < 1) nb = 1;
    it = g_occ_res.emplace(key, nb).first;
  }
  *grid = sms * it->second;
  return CMSD_OK;
}

// ---------------------------------------------------------------- workspace

constexpr size_t kAlign = 256;
size_t up(size_t x) { return (x + kAlign - 1) / kAlign * kAlign; }

struct Layout {
  size_t err, row_done, seq_word, seq_done, rec_count, res_cta_done, res_done;
  size_t rec, row_conf, row_acc, row_dstat, row_tstat, part, rpart;
  size_t total;
};

// The error word sits at offset 0 so that cmsd_workspace_errors needs no sizes;
// the two queue counters follow it (offsets 256 and 512).
Layout make_layout(int B, int K, int wmax) {
  Layout L;
  const size_t BK = (size_t)B * (size_t)K;
  size_t o = 0;
  L.err = o; o += up(sizeof(unsigned));
  L.rec_count = o; o += up(sizeof(int));
  L.res_cta_done = o; o += up(sizeof(int));
  L.row_done = o; o += up(BK * sizeof(int));
  L.seq_word = o; o += up((size_t)B * sizeof(unsigned long long));
  L.seq_done = o; o += up((size_t)B * sizeof(int));
  L.res_done = o; o += up((size_t)B * sizeof(int));
  L.rec = o; o += up((size_t)B * sizeof(int4));
  L.row_conf = o; o += up(BK * sizeof(unsigned long long));
  L.row_acc = o; o += up(BK * sizeof(int));
  L.row_dstat = o; o += up(BK * sizeof(float2));
  L.row_tstat = o; o += up(BK * sizeof(float2));
  L.part = o; o += up((BK + (size_t)wmax) * sizeof(Partial));
  L.rpart = o; o += up(((size_t)B + (size_t)wmax) * sizeof(UnitResult));
  L.total = o;
  return L;
}

Workspace carve(void* ws, const Layout& L) {
  char* p = (char*)ws;
  Workspace W;
  W.err = (unsigned*)(p + L.err);
  W.row_done = (int*)(p + L.row_done);
  W.seq_word = (unsigned long long*)(p + L.seq_word);
  W.seq_done = (int*)(p + L.seq_done);
  W.rec_count = (int*)(p + L.rec_count);
  W.res_cta_done = (int*)(p + L.res_cta_done);
  W.res_done = (int*)(p + L.res_done);
  W.rec = (int4*)(p + L.rec);
  W.row_conf = (unsigned long long*)(p + L.row_conf);
  W.row_acc = (int*)(p + L.row_acc);
  W.row_dstat = (float2*)(p + L.row_dstat);
  W.row_tstat = (float2*)(p + L.row_tstat);
  W.part = (Partial*)(p + L.part);
  W.rpart = (UnitResult*)(p + L.rpart);
  return W;
}

int wmax_warps(int* wmax) {
  int sms = 0;
  int rc = device_sms(&sms);
  if (rc) return rc;
  *wmax = sms * kMaxWarpsPerSM;
  return CMSD_OK;
}

// ---------------------------------------------------------------- timing

struct Profiler {
  bool on = false;
  int max_calls = 0;
  int n = 0;
  std::vector<cudaEvent_t> ev;   // 3 per call: start, after the streaming kernel, after the resample kernel
} g_prof;

void prof_record(int slot, cudaStream_t s) {
  if (!g_prof.on || g_prof.n >= g_prof.max_calls) return;
  cudaEventRecord(g_prof.ev[3 * g_prof.n + slot], s);
  if (slot == 2) ++g_prof.n;
}

// ---------------------------------------------------------------- checks

bool aligned16(const void* p) { return ((uintptr_t)p & 15u) == 0; }

int check_sizes(int B, int K, int V, int dtype, const int32_t* k_row) {
  if (dtype != CMSD_F32 && dtype != CMSD_BF16) return CMSD_EDTYPE;
  if (B < 0 || K < 0 || K > 1024 || V < 2) return CMSD_EINVAL;
  if ((long long)B * (long long)K > 0x7FFFFFFFLL) return CMSD_EINVAL;
  if ((double)B * (double)K * (double)V >= 70368744177664.0) return CMSD_EINVAL;   // 2^46
  if (k_row && B > kMaxRaggedB) return CMSD_EINVAL;
  return CMSD_OK;
}

int check_params(const cmsd_params* p, bool need_rule) {
  if (!p) return CMSD_EINVAL;
  if (need_rule && p->rule != CMSD_RULE_PAPER && p->rule != CMSD_RULE_SAMPLED) return CMSD_EDTYPE;
  if (p->k_min < 1 || p->k_max < p->k_min) return CMSD_EINVAL;
  float sum = 0.f;
  for (int j = 0; j < 3; ++j) {
    if (!(p->lambda[j] >= 0.f && p->lambda[j] <= 1.f)) return CMSD_EINVAL;
    sum += p->lambda[j];
  }
  if (fabsf(sum - 1.0f) > 1e-5f) return CMSD_EINVAL;
  if (!(p->beta_sig > 0.f) || !isfinite(p->beta_sig)) return CMSD_EINVAL;
  if (p->beta_rank < 0) return CMSD_EINVAL;
  if (!(p->alpha > 0.f && p->alpha <= 1.f)) return CMSD_EINVAL;
  if (!isfinite(p->tau_base) || !isfinite(p->gamma)) return CMSD_EINVAL;
  if (p->tau_sign != 1 && p->tau_sign != -1) return CMSD_EINVAL;
  if (p->k_fixed != 0 && (p->k_fixed < p->k_min || p->k_fixed > p->k_max)) return CMSD_EINVAL;
  if (p->bonus != 0 && p->bonus != 1) return CMSD_EINVAL;
  return CMSD_OK;
}

// With the bonus row the verifier tensor has K + 1 rows per sequence while the
// drafter's has K: their rows stay equally aligned only if a row is a whole
// number of 16-byte vectors.
int check_bonus_layout(const cmsd_params* p, int V, int dtype) {
  if (!p->bonus) return CMSD_OK;
  const size_t row_bytes = (size_t)V * (dtype == CMSD_F32 ? 4 : 2);
  return (row_bytes % 16) == 0 ? CMSD_OK : CMSD_EINVAL;
}

void fill_params(StreamArgs& a, const cmsd_params* p) {
  a.k_min = p->k_min;
  a.k_max = p->k_max;
  a.lam0 = p->lambda[0];
  a.lam1 = p->lambda[1];
  a.lam2 = p->lambda[2];
  a.beta_sig = p->beta_sig;
  a.beta_rank = p->beta_rank;
  a.alpha = p->alpha;
  a.tau_base = p->tau_base;
  a.gamma = p->gamma;
  a.tau_sign = p->tau_sign;
  a.k_fixed = p->k_fixed;
  a.bonus = p->bonus;
}

void fill_sizes(StreamArgs& a, int B, int K, int V) {
  a.B = B; a.K = K; a.V = V;
  a.inv_log_v = (float)(1.0 / log((double)V));
  a.soft_norm = (float)(1.0 / (1.0 - 1.0 / (double)V));
}

// CTAs per cluster that choose_seq weighs.
constexpr int kSeqSizes[] = {1, 2, 3, 4, 5, 6, 7, 8, 9, 10, 12, 16};
constexpr int kSeqNumSizes = 12;

// Clusters of seq_kernel that can be resident on device dev, which is current
// (cached; n: index into kSeqSizes).
int seq_resident(int dev, int dtype, int n, int threads) {
  static std::atomic<int> known[64][2][2][kSeqNumSizes];   // 0: not asked yet, else the answer + 1
  std::atomic<int>& k = known[dev & 63][dtype][threads == 512][n];
  int v = dev < 64 ? k.load(std::memory_order_relaxed) : 0;
  if (v == 0) {
    v = 1 + (dtype == CMSD_F32 ? seq_clusters_f32(kSeqSizes[n], threads) : seq_clusters_bf16(kSeqSizes[n], threads));
    if (dev < 64) k.store(v, std::memory_order_relaxed);
  }
  return v - 1;
}

// Which kernel takes a call: the one-launch pass with *nc CTAs of *threads
// threads per sequence (true), or the streaming kernel and its second pass.
//
// Both times are estimated, in microseconds, from what was measured on a
// GB300 over K = 1..16, V = 32000..152064, B = 1..600 (bf16; f32 alike):
//   streaming kernel   8 + bytes / 6900 MB/s, up to 3 more for ragged windows
//     (their prefix, and rows cut on the device), more when whole rows leave
//     over a tenth of the warps without one (B=80 K=8 V=128256: 67.9), and with
//     a second launch 7.5 more (11 with the bonus row), 0.015 and 0.08 per MB
//     of its row per sequence beyond 64, and 1.5 per 100000 entries where it
//     draws from rows off 16-byte boundaries (B=30 K=8 ragged verify: V=128256
//     19.7, V=128255 22.5);
//   one launch         5, a draw 3.5 (cluster_race) or 4.5 and 0.06 per KB of a
//     CTA's share beyond 64 (cluster_draw; twice the share off 16-byte
//     boundaries, where it takes over at half the share: B=10 K=1 V=152063
//     verify 11.1 by 16 CTAs of 256 threads, 9.4 raced by ten of 512; one CTA a
//     sequence, B=167 K=1 V=128255 f32 verify: 93.0, streamed 44.8), and the time of a
//     sequence's bytes through its CTAs (a CTA of 256 threads: 27 KB a
//     microsecond under the PAPER rule, 23.5 under the sampled rule, 21 for
//     the drafter alone, 30 for the target alone (33 under the PAPER rule when
//     windows are ragged, a fifth less off 16-byte boundaries); one of 512
//     twice that; a tenth more with an SM to itself, a tenth (sampled: a fifth)
//     more when both tensors' windows are ragged and neighbours end early),
//     times the waves when not
//     every cluster is resident (the draw and 3.5 more each, 10 with clusters of
//     several CTAs), and no less than the bytes at 6900 MB/s.
//
// Every cluster should be resident at once, and not all of the number that the
// occupancy query names are: clusters of 256-thread CTAs left some waiting
// above 93 in 100 of it (B=97 K=4 V=128256 by threes: 48.3 against 35.4
// streamed; B=90: 32.1), odd clusters of 512-thread CTAs, each with an SM to
// itself, near the limit (B=28 K=8 by fives: 40.7 against 33.2; B=26: 27.0),
// even ones not (SMs come in pairs).  Measured on both sides, K=8 V=128256
// sampled, streamed and in one launch: B=16 26.1, 22.6 (clusters of twelve);
// B=32 35.6, 30.2 (of eight); B=40 39.4, 38.0 (of three with 512 threads);
// B=64 54.2, 52.8 (of four).
//
// Ragged windows are unknown here: half full on average, and the longest
// decides the one-launch pass, since a sequence keeps to its cluster.  They may
// also all be full, so no more clusters count as resident than of full windows.
// A tenth more than the query names gained where windows were short (B=48 K=12
// V=32001 sampled verify, 46 clusters of six resident: 13.6, by fives 15.6,
// streamed 18.1) and lost more where they were full (22.0, 17.6, 21.5; B=38
// K=8 V=128256 sampled 49.8 by eights, 35.4 by sevens, 39.8 streamed).
//
// Over 7237 calls (K = 1 .. 16, B = 1 .. 600, V = 8000 .. 152064, ragged windows
// of a third of K on average, spread over 0..K, half or full), each timed both
// ways and with up to ten clusters, the choice takes 1.042 times the best of
// them and is slower than the streaming kernel by over 3 % at 1.0 % of them, at
// worst 1.23 times (B=96 K=12 V=8000 PAPER, whose pieces come out uneven).
//
// sms: the device's; resident(n, threads): clusters of kSeqSizes[n] such CTAs
// that it holds at once (a small partition may hold few or none of the large
// ones).
template <typename Resident>
bool choose_seq(int dtype, int mode, bool sampled, bool second, const StreamArgs& a, int sms, Resident resident, int* nc,
                int* threads) {
  if (a.K > kPackedMaxK || (second && sampled && !seq_draw_fits(dtype, a.V))) return false;
  const double kb = (double)a.K * a.V * (dtype == CMSD_F32 ? 4 : 2) * (mode == kModeFused ? 2 : 1) * 1e-3;
  const double stream = a.B * kb * (a.k_row ? 0.5 : 1.0) / 6900;
  double flat = 8 + stream;
  const int warps = sms * kStreamWarps;                           // the streaming kernel's
  if (!a.k_row && (int64_t)a.B * a.K < warps) {                   // (the rows' warps, whole rows apart from the rest)
    const double used = (double)(warps / (a.B * a.K)) * (a.B * a.K) / warps;
    if (used >= 0.75 && used < 0.9) flat += stream * 0.5 * (0.9 - used);
  }
  const int per = dtype == CMSD_F32 ? 4 : 8;             // entries per 16-byte vector
  const bool odd = a.V % per != 0;                       // rows off 16-byte boundaries
  const double row = (double)a.V * (dtype == CMSD_F32 ? 4 : 2) * 1e-3;
  if (second) {
    flat += a.bonus ? 11 : 7.5;
    if (a.B > 64) flat += (a.B - 64) * (0.015 + 8e-5 * row * (sampled && odd ? 1.5 : 1));
    if (sampled && odd) flat += 1.5e-5 * a.V;
  }
  if (a.k_row) flat += mode == kModeVerify ? 2.5 : (second && sampled && a.bonus ? 0.5 : 3);
  double rate = mode == kModeConf ? 21 : (mode == kModeVerify ? (sampled || !a.k_row ? 30 : 33) : (sampled ? 23.5 : 27));
  if (mode == kModeVerify && odd) rate *= 0.8;
  double best = 0.985 * flat;              // (a near tie stays with the streaming kernel)
  *nc = 0;
  for (int th = 256; th <= 512; th *= 2) {
    for (int k = 0; k < kSeqNumSizes; ++k) {
      const int n = kSeqSizes[k];
      // at least two 16-byte vectors per lane and piece, or more CTAs gain nothing
      if (n > 1 && kb * 1e3 < (double)n * (th / 32) * 1024 * (mode == kModeFused ? 2 : 1)) break;
      // (cluster_race: two blocks of groups per lane set, one off 16-byte boundaries)
      const bool race = a.V <= (int64_t)(odd ? 4 : 8) * n * th * per;
      double draw = second ? 3.5 : 0;
      if (second && sampled && !race) {
        const double share = row / (n * (th / 256)) * (odd ? 2 : 1);
        draw = 4.5 + (share > 64 ? 0.06 * (share - 64) : 0.0);
      }
      const double fixed = 5 + (th == 512 ? 0.7 : 0.0) + draw;
      const double full = kb / n / (rate * (th / 256));
      if (fixed + full / 1.32 >= best) continue;
      const int res = resident(k, th);
      if (res < 1) continue;
      int fit = res;
      if (th == 512 && (n & 1)) fit = res * 96 / 100;
      else if (th == 256 && n >= 3) fit = res * 93 / 100;
      if (fit < 1) fit = 1;
      const int waves = (a.B - 1) / fit + 1;
      double ease = (int64_t)a.B * n * (th / 256) <= sms ? 1.1 : 1.0;          // an SM to itself
      if (a.k_row && mode == kModeFused && waves == 1) ease *= sampled ? 1.2 : 1.1;   // neighbours that end early
      const double part = full / ease;
      const double t = fixed + (draw + (n == 1 ? 3.5 : 10.0)) * (waves - 1) +
                       (waves * part > stream ? waves * part : stream);
      if (t < best) {
        best = t;
        *nc = n;
        *threads = th;
      }
    }
  }
  return *nc > 0;
}

// Clusters of draw_kernel (nc > 0) or of the staged residual draw (nc == 0)
// that can be resident on the current device for rows of V entries (cached).
int draw_resident(int dtype, int V, int nc) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 0;
  const auto key = std::make_tuple(dev, dtype, V, nc);
  std::lock_guard<std::mutex> lk(g_mu);
  auto it = g_draw_res.find(key);
  if (it == g_draw_res.end()) {
    if (g_draw_res.size() >= 4096) g_draw_res.clear();
    int n;
    if (nc == 0) n = dtype == CMSD_F32 ? resample_bound_clusters_f32(V) : resample_bound_clusters_bf16(V);
    else n = dtype == CMSD_F32 ? draw_clusters_f32(V, nc) : draw_clusters_bf16(V, nc);
    it = g_draw_res.emplace(key, n).first;
  }
  return it->second;
}

// Which kernel makes the second pass of a streamed call, or false where a
// row's share does not fit (resample_kernel draws): the staged residual draw
// (a call without the bonus row), or draw_kernel with four CTAs per sequence,
// or with two.  Staging pays where few groups are left out by the bound (a
// target close to its drafter: each group left is read again), and costs turns
// beyond the resident clusters, fewer than draw_kernel's; both grow with a
// row's bytes (`row`; half as much again off 16-byte boundaries, where a vector
// takes two loads).  us a call at K=1, staged, four, two, for targets at drafter
// + N(0,1) and, in brackets, + N(0,1)/2 with the drafter's argmax drafted:
//   B=100 V=32000 bf16 17.5, 16.7, 17.2 (13.5, 12.7, 12.4);
//   B=100 V=128256 bf16 25.0, 26.1, 29.1 (23.5, 25.2, 27.6);
//   B=180 V=128256 bf16 33.6, 33.3, 35.4 (30.5, 32.2, 34.1);
//   B=300 V=128256 bf16 49.2, 44.4, 43.7 (41.4, 42.6, 44.1);
//   B=180 V=128255 bf16 38.0, 39.4, 46.4 (33.9, 36.7, 43.3);
//   B=300 V=128255 bf16 61.6, 51.9, 56.6 (45.4, 48.7, 54.9);
//   B=600 V=128255 bf16 109.8, 101.7, 86.5 (77.8, 74.0, 80.4);
//   B=40 V=128255 f32 (36 staged clusters resident) 27.5, 35.3, 48.9.
// Over 1070 such calls (V = 8001 .. 152064, K = 1 .. 24, four recipes) the
// choice takes 1.006 times the best of the three (always staged 1.068, by the
// number of sequences alone 1.033), and at worst 1.17 times the staged draw
// (B=600 K=1 V=152063 f32).  The bonus row's race costs more per turn (four, two:
// B=130 V=128256 bf16 30.4, 34.3, B=152 39.3, 36.5); its argmax under the PAPER
// rule is one round of loads (B=450 V=128256 50.5, 55.1; V=32000 23.9, 23.4).
// resident(nc): clusters of draw_kernel (nc > 0) or of the staged draw (0)
// that the device holds at once.
struct DrawPlan {
  int clusters, nc;                        // nc == 0: the staged residual draw
};
template <typename Resident>
bool draw_plan(int dtype, bool sampled, bool bonus, int B, int V, Resident resident, DrawPlan* d) {
  const int es = dtype == CMSD_F32 ? 4 : 2;
  const bool odd = (int64_t)V * es % 16 != 0;
  const int64_t row = (int64_t)V * es * (odd ? 3 : 2) / 2;
  const bool wide = row >= 290000, mid = row >= 140000;
  const int64_t staged = sampled && !bonus ? resident(0) : 0;
  int res = (int)staged;
  d->nc = 0;
  if (B > staged * (wide ? (odd ? 15 : 10) : (mid ? 7 : 5)) / 5) {
    d->nc = 4;
    res = resident(4);
    int64_t most = res;                    // sequences with four CTAs each
    if (!sampled) most = mid ? B : res;
    else if (!bonus) most = (int64_t)res * (wide ? (odd ? 62 : 42) : (mid ? 40 : 21)) / 20;
    const int two = B > most ? resident(2) : 0;      // (0: half a row's groups do not fit)
    if (two > 0) {
      d->nc = 2;
      res = two;
    }
  }
  d->clusters = B < 2 * res ? B : 2 * res;
  return res > 0;
}
bool draw_plan(int dtype, bool sampled, bool bonus, int B, int V, DrawPlan* d) {
  return draw_plan(dtype, sampled, bonus, B, V, [&](int nc) { return draw_resident(dtype, V, nc); }, d);
}

cudaError_t launch_draw(int dtype, bool sampled, const StreamArgs& a, const DrawPlan& d, cudaStream_t s) {
  if (d.nc == 0)
    return dtype == CMSD_F32 ? launch_resample_bound_f32(a, d.clusters, s) : launch_resample_bound_bf16(a, d.clusters, s);
  return dtype == CMSD_F32 ? launch_draw_f32(sampled, a, d.clusters, d.nc, s)
                           : launch_draw_bf16(sampled, a, d.clusters, d.nc, s);
}

// The current device's choice for a call: *nc CTAs of *threads threads per
// sequence, or *nc = 0 for the streaming kernel.
int choose(int dtype, int mode, bool sampled, bool second, const StreamArgs& a, int* nc, int* threads) {
  int dev = 0, sms = 0;
  const cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return cuda_fail(e);
  const int rc = device_sms(&sms);
  if (rc) return rc;
  *nc = *threads = 0;
  if (!choose_seq(dtype, mode, sampled, second, a, sms, [&](int n, int th) { return seq_resident(dev, dtype, n, th); },
                  nc, threads))
    *nc = *threads = 0;
  return CMSD_OK;
}

// Threads per CTA of the streaming kernel: kStreamThreads, but for short rows
// that its warps' slices would cross the ends of (more rows than warps, or too
// few of the warps used by whole pieces of a row).  There each row ends a
// warp's pipeline and reduction, and more warps with shorter stages hide it:
// 768 threads and two vectors against 512 and four, at 2880 rows (whole rows
// again with 768) V=4000 sampled 0.82 of the time, V=16000 0.92, V=64128 0.96,
// V=128256 1.03; at 7200 (crossed by both) V=8000 0.84, V=32000 0.90, V=50257
// 0.96; PAPER at 816 rows V=4000 0.68 (14.7 against 21.6 us), V=32000 0.94; the
// drafter alone at 7200 V=8000 0.92, V=32000 1.04.  Rows in whole pieces lose
// 1 to 39 per cent by it (V=4000 at 2400 rows 1.23).  f32 rows gain at half the
// length (V=8000 0.94, V=32000 0.98 at 2880 rows).  Ragged windows count half
// their rows.
int stream_threads(int dtype, int mode, bool sampled, const StreamArgs& a, int sms) {
  const int64_t rows64 = (int64_t)a.B * a.K;
  const int rows = (int)(a.k_row ? (rows64 + 1) / 2 : rows64);
  const int vec = dtype == CMSD_F32 ? 4 : 8;
  const int64_t min_len = stream_min_len(a.V);
  if (StreamSplit(rows, a.V, vec, sms * (kStreamThreads / 32), min_len).wpr > 0) return kStreamThreads;
  const bool whole = StreamSplit(rows, a.V, vec, sms * (kStreamThreadsShort / 32), min_len).wpr > 0;
  int most;                                // entries of a bf16 row, in thousands
  if (mode == kModeConf) most = whole ? 20 : 10;
  else if (mode == kModeVerify) most = whole ? 65 : 33;
  else most = sampled ? (whole ? 65 : 55) : (whole ? 33 : 20);
  return (int64_t)a.V * (dtype == CMSD_F32 ? 4 : 1) <= most * 1000ll ? kStreamThreadsShort : kStreamThreads;
}

// (nc > 0: the one-launch kernel with that many CTAs of `threads` threads per
// sequence, whatever the rule says)
int launch(int dtype, int mode, bool sampled, StreamArgs& a, void* ws, size_t ws_bytes,
           cudaStream_t s, int nc = 0, int threads = 0) {
  int wmax = 0;
  int rc = wmax_warps(&wmax);
  if (rc) return rc;
  const Layout L = make_layout(a.B, a.K, wmax);
  if (!ws || ws_bytes < L.total) return CMSD_ENOWS;
  a.ws = carve(ws, L);
  const bool bonus = mode != kModeConf && a.bonus;
  a.Kt = bonus ? a.K + 1 : a.K;
  a.Ko = bonus ? a.K + 1 : a.K;
  const bool second = mode != kModeConf && (sampled || bonus);
  if (nc == 0) {
    rc = choose(dtype, mode, sampled, second, a, &nc, &threads);
    if (rc) return rc;
  }
  if (nc > 0) {
    prof_record(0, s);
    const cudaError_t e = dtype == CMSD_F32 ? launch_seq_f32(mode, sampled, second, a, nc, threads, s)
                                            : launch_seq_bf16(mode, sampled, second, a, nc, threads, s);
    if (e != cudaSuccess) return cuda_fail(e);
    prof_record(1, s);
    prof_record(2, s);
    return CMSD_OK;
  }
  const size_t smem = stream_smem_bytes(a.B, a.k_row != nullptr);
  int grid = 0;
  int sms = 0;
  rc = device_sms(&sms);
  if (rc) return rc;
  const int st = stream_threads(dtype, mode, sampled, a, sms);
  rc = stream_grid(dtype, mode, sampled, second, st, smem, &grid);
  if (rc) return rc;
  int g2 = 0;
  DrawPlan dp;
  const bool bound = second && draw_plan(dtype, sampled, bonus, a.B, a.V, &dp);
  if (second && !bound) {
    rc = resample_grid(dtype, sampled, &g2);
    if (rc) return rc;
  }
  a.nwarps = grid * (st / 32);
  if (!a.k_row) a.split = StreamSplit(a.B * a.K, a.V, dtype == CMSD_F32 ? 4 : 8, a.nwarps, stream_min_len(a.V));
  a.rec_by_seq = bound ? 1 : 0;
  prof_record(0, s);
  cudaError_t e = dtype == CMSD_F32 ? launch_stream_f32(mode, sampled, second, a, grid, st, smem, s)
                                    : launch_stream_bf16(mode, sampled, second, a, grid, st, smem, s);
  if (e != cudaSuccess) return cuda_fail(e);
  prof_record(1, s);
  if (second) {
    StreamArgs b = a;
    b.nwarps = g2 * kResWarps;
    if (bound)
      e = launch_draw(dtype, sampled, b, dp, s);
    else
      e = dtype == CMSD_F32 ? launch_resample_f32(sampled, b, g2, s) : launch_resample_bf16(sampled, b, g2, s);
    if (e != cudaSuccess) {
      // the streaming kernel has queued rows that no resample kernel will
      // drain: return the queue counters to zero so the workspace stays usable
      cudaMemsetAsync(a.ws.rec_count, 0, sizeof(int), s);
      cudaMemsetAsync(a.ws.res_cta_done, 0, sizeof(int), s);
      if (bound) cudaMemsetAsync(a.ws.rec, 0, (size_t)a.B * sizeof(int4), s);   // the released record words
      return cuda_fail(e);
    }
  }
  prof_record(2, s);
  return CMSD_OK;
}

StreamArgs blank_args() {
  StreamArgs a;
  memset(&a, 0, sizeof(a));
  return a;
}

}  // namespace

namespace cmsd {

// Every host-side check of cmsd_confidence_verify (sizes, parameters, bonus
// layout, required pointers, alignment), without launching anything.
int validate_fused(const void* draft_logits, const void* target_logits, const int32_t* draft_tokens,
                   const int32_t* k_row, int B, int K, int V, int dtype, const void* params,
                   const int32_t* n_accept, const int32_t* out_tokens) {
  const cmsd_params* p = (const cmsd_params*)params;
  int rc = check_sizes(B, K, V, dtype, k_row);
  if (rc) return rc;
  rc = check_params(p, true);
  if (rc) return rc;
  rc = check_bonus_layout(p, V, dtype);
  if (rc) return rc;
  if (B == 0 || K == 0) return CMSD_OK;
  if (!draft_logits || !target_logits || !draft_tokens || !n_accept || !out_tokens) return CMSD_EINVAL;
  if (!aligned16(draft_logits) || !aligned16(target_logits)) return CMSD_EALIGN;
  return CMSD_OK;
}

}  // namespace cmsd

// ============================================================ C ABI

// ---------------------------------------------------------------- LM head

namespace {
struct LmLayout {
  size_t row_conf, part, total;
  int nct, nb;
};
int lm_layout(int R, int V, LmLayout* L) {
  int sms = 0;
  int rc = device_sms(&sms);
  if (rc) return rc;
  L->nct = lmhead_ctas_per_block(sms, R, V);
  L->nb = lmhead_block_rows(R);
  const size_t nrb = (size_t)(R + L->nb - 1) / L->nb;
  size_t o = up(sizeof(unsigned));
  L->row_conf = o; o += up((size_t)R * sizeof(unsigned long long));
  L->part = o; o += up(nrb * (size_t)L->nct * L->nb * sizeof(Partial));
  L->total = o;
  return CMSD_OK;
}
int check_lmhead(int R, int d, int V) {
  if (R < 0 || d < 64 || d % 64 != 0 || d > (1 << 20) || V < 2) return CMSD_EINVAL;
  if ((double)R * (double)V >= 70368744177664.0) return CMSD_EINVAL;   // 2^46 logits
  return CMSD_OK;
}
}  // namespace

extern "C" {

void cmsd_params_default(cmsd_params* p, int K, int rule) {
  if (!p) return;
  p->k_min = 1;
  p->k_max = K > 0 ? K : 1;
  p->lambda[0] = p->lambda[1] = p->lambda[2] = 1.0f / 3.0f;
  p->beta_sig = 1.0f;
  p->beta_rank = rule == CMSD_RULE_SAMPLED ? 0 : 3;
  p->alpha = 1.0f;
  p->tau_base = 0.1f;
  p->gamma = 1.0f;
  p->tau_sign = 1;
  p->rule = rule;
  p->k_fixed = 0;
  p->bonus = 0;
}

int cmsd_params_preset(cmsd_params* p, int K, int rule, int preset) {
  if (!p) return CMSD_EINVAL;
  cmsd_params_default(p, K, rule);
  switch (preset) {
    case CMSD_PRESET_FULL: break;
    case CMSD_PRESET_FIXED_K: p->k_fixed = p->k_max; break;
    case CMSD_PRESET_FIXED_TAU: p->gamma = 0.0f; break;
    case CMSD_PRESET_FIXED_K_TAU: p->k_fixed = p->k_max; p->gamma = 0.0f; break;
    case CMSD_PRESET_ENTROPY_ONLY: p->lambda[0] = 1.0f; p->lambda[1] = p->lambda[2] = 0.0f; break;
    case CMSD_PRESET_MARGIN_ONLY: p->lambda[1] = 1.0f; p->lambda[0] = p->lambda[2] = 0.0f; break;
    case CMSD_PRESET_SOFTMAX_ONLY: p->lambda[2] = 1.0f; p->lambda[0] = p->lambda[1] = 0.0f; break;
    default: return CMSD_EINVAL;
  }
  return CMSD_OK;
}


size_t cmsd_lmhead_workspace_bytes(int R, int d, int V) {
  if (check_lmhead(R, d, V)) return 0;
  LmLayout L;
  if (lm_layout(R, V, &L)) return 0;
  return L.total;
}

int cmsd_lmhead_confidence(const void* hidden, const void* weight, int R, int d, int V,
                           const cmsd_params* p, float* H, float* margin, int32_t* argmax, float* conf,
                           float* lse, float* logits, void* ws, size_t ws_bytes, void* stream) {
  int rc = check_lmhead(R, d, V);
  if (rc) return rc;
  rc = check_params(p, false);
  if (rc) return rc;
  if (R == 0) return CMSD_OK;
  if (!hidden || !weight) return CMSD_EINVAL;
  if (!aligned16(hidden) || !aligned16(weight)) return CMSD_EALIGN;
  LmLayout L;
  rc = lm_layout(R, V, &L);
  if (rc) return rc;
  if (!ws || ws_bytes < L.total) return CMSD_ENOWS;
  StreamArgs a = blank_args();
  fill_sizes(a, R, 1, V);
  fill_params(a, p);
  a.Kt = a.Ko = 1;
  a.H = H; a.margin = margin; a.argmax = argmax; a.conf = conf; a.lse = lse;
  char* w = (char*)ws;
  a.ws.err = (unsigned*)w;
  a.ws.row_conf = (unsigned long long*)(w + L.row_conf);
  LmHeadArgs h;
  h.hidden = (const uint16_t*)hidden;
  h.weight = (const uint16_t*)weight;
  h.R = R; h.d = d; h.V = V;
  h.nct = L.nct;
  h.nb = L.nb;
  h.logits = logits;
  h.part = (Partial*)(w + L.part);
  h.err = a.ws.err;
  cudaError_t e = launch_lmhead(h, a, (cudaStream_t)stream);
  return e == cudaSuccess ? CMSD_OK : cuda_fail(e);
}

size_t cmsd_workspace_bytes(int B, int K, int V) {
  if (B < 0 || K < 0 || V < 2) return 0;
  int wmax = 0;
  if (wmax_warps(&wmax)) return 0;
  return make_layout(B, K, wmax).total;
}

int cmsd_workspace_init(void* ws, size_t ws_bytes, void* stream) {
  if (!ws || ws_bytes == 0) return CMSD_ENOWS;
  cudaError_t e = cudaMemsetAsync(ws, 0, ws_bytes, (cudaStream_t)stream);
  return e == cudaSuccess ? CMSD_OK : cuda_fail(e);
}

int cmsd_workspace_errors(void* ws, size_t ws_bytes, void* stream, uint32_t* flags_out) {
  if (!ws || ws_bytes < sizeof(unsigned) || !flags_out) return CMSD_EINVAL;
  unsigned h = 0;
  cudaStream_t s = (cudaStream_t)stream;
  cudaError_t e = cudaMemcpyAsync(&h, ws, sizeof(unsigned), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaMemsetAsync(ws, 0, sizeof(unsigned), s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return cuda_fail(e);
  *flags_out = h;
  return CMSD_OK;
}

int cmsd_test_record_wait_timeout(const void* draft_logits, const void* target_logits, int B, int K, int V,
                                  int dtype, int32_t* out_tokens, void* ws, size_t ws_bytes, void* stream) {
  int rc = check_sizes(B, K, V, dtype, nullptr);
  if (rc) return rc;
  if (B == 0 || K == 0) return CMSD_OK;
  if (!draft_logits || !target_logits || !out_tokens) return CMSD_EINVAL;
  if (!aligned16(draft_logits) || !aligned16(target_logits)) return CMSD_EALIGN;
  DrawPlan dp;
  if (!draw_plan(dtype, true, false, B, V, &dp)) return CMSD_EDTYPE;
  int wmax = 0;
  rc = wmax_warps(&wmax);
  if (rc) return rc;
  const Layout L = make_layout(B, K, wmax);
  if (!ws || ws_bytes < L.total) return CMSD_ENOWS;
  StreamArgs a = blank_args();
  fill_sizes(a, B, K, V);
  a.draft = draft_logits;
  a.target = target_logits;
  a.out_tokens = out_tokens;
  a.Kt = a.Ko = K;
  a.rec_by_seq = 1;
  a.ws = carve(ws, L);
  cudaStream_t s = (cudaStream_t)stream;
  // no record is released: every sequence's wait runs out
  cudaError_t e = cudaMemsetAsync(a.ws.rec, 0, (size_t)B * sizeof(int4), s);
  if (e != cudaSuccess) return cuda_fail(e);
  e = launch_draw(dtype, true, a, dp, s);
  return e == cudaSuccess ? CMSD_OK : cuda_fail(e);
}

int cmsd_test_choose(int call, int B, int K, int V, int dtype, int rule, int bonus, int ragged, int sms,
                     const int32_t* resident, int32_t* cluster, int32_t* threads) {
  const int32_t some = 0;
  const int rc = check_sizes(B, K, V, dtype, ragged ? &some : nullptr);
  if (rc) return rc;
  if (call < kModeConf || call > kModeFused || B < 1 || K < 1 || sms < 1 || !resident || !cluster || !threads) return CMSD_EINVAL;
  StreamArgs a = blank_args();
  fill_sizes(a, B, K, V);
  a.bonus = bonus != 0;
  a.k_row = ragged ? &some : nullptr;
  const bool sampled = call != kModeConf && rule == CMSD_RULE_SAMPLED;
  int nc = 0, th = 0;
  choose_seq(dtype, call, sampled, call != kModeConf && (sampled || bonus), a, sms,
             [&](int n, int t) { return (int)resident[(t == 512 ? 17 : 0) + kSeqSizes[n]]; }, &nc, &th);
  *cluster = nc;
  *threads = nc > 0 ? th : stream_threads(dtype, call, sampled, a, sms);
  return CMSD_OK;
}

int cmsd_test_draw(int B, int V, int dtype, int rule, int bonus, const int32_t* resident, int32_t* ctas) {
  const int rc = check_sizes(B, 1, V, dtype, nullptr);
  if (rc) return rc;
  if (B < 1 || !resident || !ctas || (rule != CMSD_RULE_SAMPLED && !bonus)) return CMSD_EINVAL;
  DrawPlan d;
  const bool fits = draw_plan(dtype, rule == CMSD_RULE_SAMPLED, bonus != 0, B, V,
                              [&](int nc) { return (int)resident[nc == 0 ? 0 : (nc == 4 ? 1 : 2)]; }, &d);
  *ctas = fits ? d.nc : -1;
  return CMSD_OK;
}

int cmsd_test_confidence_verify_cluster(const void* draft_logits, const void* target_logits,
                                        const int32_t* draft_tokens, const int32_t* k_row, int B, int K, int V,
                                        int dtype, const cmsd_params* p, uint64_t seed, uint32_t iteration, float* H,
                                        float* margin, int32_t* argmax, float* conf, float* lse, int32_t* k_next,
                                        int32_t* n_accept, int32_t* out_tokens, uint8_t* accept, void* ws,
                                        size_t ws_bytes, void* stream, int cluster, int threads) {
  const int rc = validate_fused(draft_logits, target_logits, draft_tokens, k_row, B, K, V, dtype, p,
                                n_accept, out_tokens);
  if (rc) return rc;
  if (B == 0 || K == 0) return CMSD_OK;
  const bool sampled = p->rule == CMSD_RULE_SAMPLED;
  int size = -1, dev = 0;
  for (int n = 0; n < kSeqNumSizes; ++n)
    if (kSeqSizes[n] == cluster) size = n;
  if (size < 0 || (threads != 256 && threads != 512) || K > kPackedMaxK || (sampled && !seq_draw_fits(dtype, V)))
    return CMSD_EDTYPE;
  const cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return cuda_fail(e);
  if (seq_resident(dev, dtype, size, threads) < 1) return CMSD_EDTYPE;
  StreamArgs a = blank_args();
  a.draft = draft_logits;
  a.target = target_logits;
  a.tokens = draft_tokens;
  a.k_row = k_row;
  fill_sizes(a, B, K, V);
  fill_params(a, p);
  a.seed = seed;
  a.iteration = iteration;
  a.H = H; a.margin = margin; a.argmax = argmax; a.conf = conf; a.lse = lse; a.k_next = k_next;
  a.n_accept = n_accept; a.out_tokens = out_tokens; a.accept = accept;
  return launch(dtype, kModeFused, sampled, a, ws, ws_bytes, (cudaStream_t)stream, cluster, threads);
}

int cmsd_confidence(const void* draft_logits, int B, int K, int V, int dtype, const int32_t* k_row,
                    const cmsd_params* p, float* H, float* margin, int32_t* argmax, float* conf,
                    float* lse, int32_t* k_next, void* ws, size_t ws_bytes, void* stream) {
  int rc = check_sizes(B, K, V, dtype, k_row);
  if (rc) return rc;
  rc = check_params(p, false);
  if (rc) return rc;
  if (B == 0 || K == 0) return CMSD_OK;
  if (!draft_logits) return CMSD_EINVAL;
  if (!aligned16(draft_logits)) return CMSD_EALIGN;
  StreamArgs a = blank_args();
  a.draft = draft_logits;
  a.k_row = k_row;
  fill_sizes(a, B, K, V);
  fill_params(a, p);
  a.H = H; a.margin = margin; a.argmax = argmax; a.conf = conf; a.lse = lse; a.k_next = k_next;
  return launch(dtype, kModeConf, false, a, ws, ws_bytes, (cudaStream_t)stream);
}

int cmsd_verify(const void* draft_logits, const void* target_logits, const int32_t* draft_tokens,
                const int32_t* k_row, int B, int K, int V, int dtype, const cmsd_params* p,
                const float* conf, const float* draft_lse, uint64_t seed, uint32_t iteration,
                int32_t* n_accept, int32_t* out_tokens, uint8_t* accept, void* ws, size_t ws_bytes,
                void* stream) {
  int rc = check_sizes(B, K, V, dtype, k_row);
  if (rc) return rc;
  rc = check_params(p, true);
  if (rc) return rc;
  rc = check_bonus_layout(p, V, dtype);
  if (rc) return rc;
  if (B == 0 || K == 0) return CMSD_OK;
  const bool sampled = p->rule == CMSD_RULE_SAMPLED;
  if (!draft_logits || !target_logits || !draft_tokens || !conf || !n_accept || !out_tokens)
    return CMSD_EINVAL;
  if (sampled && !draft_lse) return CMSD_EINVAL;
  if (!aligned16(draft_logits) || !aligned16(target_logits)) return CMSD_EALIGN;
  StreamArgs a = blank_args();
  a.draft = draft_logits;
  a.target = target_logits;
  a.tokens = draft_tokens;
  a.k_row = k_row;
  fill_sizes(a, B, K, V);
  fill_params(a, p);
  a.seed = seed;
  a.iteration = iteration;
  a.conf_in = conf;
  a.lse_in = draft_lse;
  a.n_accept = n_accept; a.out_tokens = out_tokens; a.accept = accept;
  return launch(dtype, kModeVerify, sampled, a, ws, ws_bytes, (cudaStream_t)stream);
}

int cmsd_confidence_verify(const void* draft_logits, const void* target_logits,
                           const int32_t* draft_tokens, const int32_t* k_row, int B, int K, int V,
                           int dtype, const cmsd_params* p, uint64_t seed, uint32_t iteration,
                           float* H, float* margin, int32_t* argmax, float* conf, float* lse,
                           int32_t* k_next, int32_t* n_accept, int32_t* out_tokens, uint8_t* accept,
                           void* ws, size_t ws_bytes, void* stream) {
  const int rc = validate_fused(draft_logits, target_logits, draft_tokens, k_row, B, K, V, dtype, p,
                                n_accept, out_tokens);
  if (rc) return rc;
  if (B == 0 || K == 0) return CMSD_OK;
  const bool sampled = p->rule == CMSD_RULE_SAMPLED;
  StreamArgs a = blank_args();
  a.draft = draft_logits;
  a.target = target_logits;
  a.tokens = draft_tokens;
  a.k_row = k_row;
  fill_sizes(a, B, K, V);
  fill_params(a, p);
  a.seed = seed;
  a.iteration = iteration;
  a.H = H; a.margin = margin; a.argmax = argmax; a.conf = conf; a.lse = lse; a.k_next = k_next;
  a.n_accept = n_accept; a.out_tokens = out_tokens; a.accept = accept;
  return launch(dtype, kModeFused, sampled, a, ws, ws_bytes, (cudaStream_t)stream);
}

uint32_t cmsd_philox_u32(uint64_t seed, uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3, int word) {
  const U4 w = philox4x32_10(U4{c0, c1, c2, c3}, seed_lo(seed), seed_hi(seed));
  switch (word & 3) {
    case 0: return w.x;
    case 1: return w.y;
    case 2: return w.z;
    default: return w.w;
  }
}

int cmsd_philox_fill(uint64_t seed, uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3, uint32_t* out,
                     size_t n, void* stream) {
  if (n == 0) return CMSD_OK;
  if (!out) return CMSD_EINVAL;
  cudaError_t e = launch_philox_fill(seed, c0, c1, c2, c3, out, n, (cudaStream_t)stream);
  return e == cudaSuccess ? CMSD_OK : cuda_fail(e);
}

int cmsd_profile_start(int max_calls) {
  if (max_calls < 0) return CMSD_EINVAL;
  const size_t need = (size_t)max_calls * 3;
  while (g_prof.ev.size() < need) {
    cudaEvent_t e;
    cudaError_t err = cudaEventCreate(&e);
    if (err != cudaSuccess) return cuda_fail(err);
    g_prof.ev.push_back(e);
  }
  g_prof.on = true;
  g_prof.max_calls = max_calls;
  g_prof.n = 0;
  return CMSD_OK;
}

int cmsd_profile_stop(float* stream_ms, float* resample_ms, int max_out, int* n_out) {
  g_prof.on = false;
  const int n = g_prof.n < max_out ? g_prof.n : max_out;
  for (int j = 0; j < n; ++j) {
    cudaError_t e = cudaEventSynchronize(g_prof.ev[3 * j + 2]);
    if (e != cudaSuccess) return cuda_fail(e);
    float x = 0.f, y = 0.f;
    e = cudaEventElapsedTime(&x, g_prof.ev[3 * j], g_prof.ev[3 * j + 1]);
    if (e == cudaSuccess) e = cudaEventElapsedTime(&y, g_prof.ev[3 * j + 1], g_prof.ev[3 * j + 2]);
    if (e != cudaSuccess) return cuda_fail(e);
    if (stream_ms) stream_ms[j] = x;
    if (resample_ms) resample_ms[j] = y;
  }
  if (n_out) *n_out = n;
  g_prof.n = 0;
  return CMSD_OK;
}

int cmsd_launch_plan(int call, int B, int K, int V, int dtype, const cmsd_params* p, int ragged, int* launches,
                     int* cluster, int* threads) {
  const int32_t some = 0;
  int rc = check_sizes(B, K, V, dtype, ragged ? &some : nullptr);
  if (rc) return rc;
  if (call < kModeConf || call > kModeFused) return CMSD_EINVAL;
  rc = check_params(p, call != kModeConf);
  if (rc) return rc;
  if (call != kModeConf) {
    rc = check_bonus_layout(p, V, dtype);
    if (rc) return rc;
  }
  int nl = 0, nc = 0, th = 0;
  if (B > 0 && K > 0) {
    StreamArgs a = blank_args();
    fill_sizes(a, B, K, V);
    fill_params(a, p);
    a.k_row = ragged ? &some : nullptr;
    const bool sampled = call != kModeConf && p->rule == CMSD_RULE_SAMPLED;
    const bool second = call != kModeConf && (sampled || a.bonus);
    rc = choose(dtype, call, sampled, second, a, &nc, &th);
    if (rc) return rc;
    nl = nc > 0 || !second ? 1 : 2;
    if (nc == 0) {
      int sms = 0;
      rc = device_sms(&sms);
      if (rc) return rc;
      th = stream_threads(dtype, call, sampled, a, sms);
    }
  }
  if (launches) *launches = nl;
  if (cluster) *cluster = nc;
  if (threads) *threads = th;
  return CMSD_OK;
}

int cmsd_launch_info(int dtype, int* warps_out, int* sms_out) {
  if (dtype != CMSD_F32 && dtype != CMSD_BF16) return CMSD_EDTYPE;
  int sms = 0, grid = 0;
  int rc = device_sms(&sms);
  if (rc) return rc;
  rc = stream_grid(dtype, kModeFused, true, true, kStreamThreads, stream_smem_bytes(0, false), &grid);
  if (rc) return rc;
  if (warps_out) *warps_out = grid * kStreamWarps;
  if (sms_out) *sms_out = sms;
  return CMSD_OK;
}

const char* cmsd_strerror(int code) {
  switch (code) {
    case CMSD_OK: return "ok";
    case CMSD_EINVAL: return "invalid argument";
    case CMSD_EDTYPE: return "unknown dtype or rule";
    case CMSD_ECUDA: return "CUDA runtime error";
    case CMSD_ENOWS: return "workspace missing or too small";
    case CMSD_EALIGN: return "logit pointer not 16-byte aligned";
    case CMSD_ESCRATCH: return "problem too large for the static scratch (CMSD_STATIC_SCRATCH_BYTES)";
    default: return "unknown error";
  }
}

int cmsd_last_cuda_error(void) { return g_last_cuda; }

}  // extern "C"
