// Device generator of the decode-loop simulation's synthetic logits
// (include/cmsd_workload.h).  Input generation only: bit-identical to the
// host recipe (table lookups and IEEE float adds/multiplies with no
// contraction), so the CPU oracle can regenerate the same rows.
#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "cmsd_philox.cuh"
#include "cmsd_workload.h"

namespace cg = cooperative_groups;

namespace {

constexpr uint32_t kGenDNoise = 0xC0000002u;
constexpr uint32_t kGenTNoise = 0xC0000003u;
constexpr uint32_t kGenSpike = 0xC0000004u;
// A row is made by a cluster of kParts CTAs (most slots of a window are idle).
// One CTA of 1024 threads per row left a second wave of a few rows on 152 SMs
// and staged the table with one entry per load: 160 rows of 32000 took 21.6 us.
// Two parts of 512 threads took 17.5, four of 256 16.4, and with vector loads
// of the table 15.8.  Two 16-byte stores per thread left every store of a
// warp writing half sectors; with 32-byte stores, and the active slots first,
// 13.5 (32 windows of 5 rows on average, 41 MB written).
constexpr int kParts = 4;
constexpr int kThreads = 256;
constexpr int kTableBits = 13;   // the normal table: 2^13 float32, staged in shared memory

// The table entry that a 16-bit half of a word names by its top bits.
__device__ __forceinline__ float table_at(const float* table, uint32_t word, int half) {
  constexpr uint32_t mask = ((1u << kTableBits) - 1) << 2;               // byte offsets
  const uint32_t at = (half ? word >> (30 - kTableBits) : word >> (14 - kTableBits)) & mask;
  return *reinterpret_cast<const float*>(reinterpret_cast<const char*>(table) + at);
}

// 32 bytes, one whole sector, in one store (p on a 32-byte boundary).
__device__ __forceinline__ void store8(float* p, const float (&x)[8]) {
  asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "f"(x[0]), "f"(x[1]), "f"(x[2]),
               "f"(x[3]), "f"(x[4]), "f"(x[5]), "f"(x[6]), "f"(x[7])
               : "memory");
}

// One cluster per (b, i) slot of the [B][Kt] verifier layout, from slot0 on.
// SINGLE: rows that no vector store fits.  Eight stores of a thread's own eight
// logits touch a sector each (B=32 K=16 V=31999 51.9 us); a warp's 256 go through
// shared memory first and leave as whole lines (16.4 us).
template <bool SINGLE>
__global__ void __launch_bounds__(kThreads) __cluster_dims__(kParts, 1, 1) gen_rows_kernel(const float* __restrict__ table,
                                                            const float* __restrict__ heights_it,
                                                            uint32_t it, int slot0, int B, int K_max, int Kt, int V,
                                                            const int32_t* __restrict__ k_row,
                                                            uint32_t k0, uint32_t k1, float* draft,
                                                            float* target, int32_t* tokens) {
  // a programmatic dependent of what precedes it: placed early, reads and
  // writes nothing before that has completed
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int cluster = blockIdx.x / kParts, part = blockIdx.x - cluster * kParts;
  const int slot = slot0 + cluster;
  const int i = slot / B;                       // position-major: the idle slots come last
  const int b = slot - i * B;
  int k = K_max;
  if (k_row) {
    k = k_row[b];
    k = k < 0 ? 0 : (k > K_max ? K_max : k);
  }
  const bool has_draft = i < k;
  if (!has_draft && i >= k + (Kt - K_max)) return;
  __shared__ __align__(16) float s_table[1 << kTableBits];
  if (((uintptr_t)table & 15) == 0) {
    const float4* t4 = reinterpret_cast<const float4*>(table);
#pragma unroll
    for (int j = 0; j < (1 << kTableBits) / 4 / kThreads; ++j)
      reinterpret_cast<float4*>(s_table)[j * kThreads + threadIdx.x] = __ldg(t4 + j * kThreads + threadIdx.x);
  } else {
    for (int j = threadIdx.x; j < (1 << kTableBits); j += kThreads) s_table[j] = table[j];
  }
  __syncthreads();
  const int row = b * (K_max + 1) + i;          // generator row id
  const float h = heights_it[b];
  const cmsd::U4 sw = cmsd::philox4x32_10(cmsd::U4{0u, (uint32_t)row, it, kGenSpike}, k0, k1);
  const int spike = (int)(((uint64_t)sw.x * (uint64_t)V) >> 32);
  float* dz = draft + ((size_t)b * K_max + i) * V;
  float* tz = target + ((size_t)b * Kt + i) * V;

  float best = -__int_as_float(0x7F800000);
  int bidx = 0x7FFFFFFF;
  const int ngrp = (V + 7) / 8;
  // rows start on 32-byte boundaries when V is a multiple of 8 and the tensors
  // do: each thread then writes its 8 logits in one store; on 16-byte ones when
  // V is a multiple of 4 and the tensors do: two stores
  const bool vec8 = (V & 7) == 0 && ((((uintptr_t)draft) | ((uintptr_t)target)) & 31) == 0;
  __shared__ __align__(16) float s_out[SINGLE ? kThreads / 32 : 1][SINGLE ? 256 : 1];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  // (SINGLE: whole warps, a lane past the last group makes one that is not written)
  for (int g = part * kThreads + threadIdx.x; (SINGLE ? g - lane : g) < ngrp; g += kParts * kThreads) {
    const cmsd::U4 wd = cmsd::philox4x32_10(cmsd::U4{(uint32_t)g, (uint32_t)row, it, kGenDNoise}, k0, k1);
    const cmsd::U4 wt = cmsd::philox4x32_10(cmsd::U4{(uint32_t)g, (uint32_t)row, it, kGenTNoise}, k0, k1);
    const uint32_t dw[4] = {wd.x, wd.y, wd.z, wd.w}, tw[4] = {wt.x, wt.y, wt.z, wt.w};
    float zs[8], ts[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int v = 8 * g + j;
      float z = table_at(s_table, dw[j >> 1], j & 1);
      if (v == spike) z = __fadd_rn(z, h);
      zs[j] = z;
      ts[j] = __fadd_rn(z, __fmul_rn(0.8f, table_at(s_table, tw[j >> 1], j & 1)));
    }
    float m = -__int_as_float(0x7F800000);       // the group's maximum and its lowest place
    int mj = 0;
#pragma unroll
    for (int j = 7; j >= 0; --j)
      if (8u * (uint32_t)g + j < (uint32_t)V && zs[j] >= m) { m = zs[j]; mj = j; }
    if (m > best) { best = m; bidx = 8 * g + mj; }
    if (SINGLE) {
      auto put = [&](float* row_at, const float (&x)[8]) {
        float4* out = reinterpret_cast<float4*>(s_out[warp] + 8 * lane);
        __syncwarp();
        out[0] = make_float4(x[0], x[1], x[2], x[3]);
        out[1] = make_float4(x[4], x[5], x[6], x[7]);
        __syncwarp();
        const uint32_t v0 = 8u * (uint32_t)(g - lane) + (uint32_t)lane;
#pragma unroll
        for (int j = 0; j < 8; ++j)
          if (v0 + 32u * j < (uint32_t)V) row_at[v0 + 32u * j] = s_out[warp][lane + 32 * j];
      };
      if (has_draft) put(dz, zs);
      put(tz, ts);
    } else if (vec8) {
      if (has_draft) store8(dz + 8 * g, zs);
      store8(tz + 8 * g, ts);
    } else if (8 * g + 8 <= V) {
      float4* d4 = reinterpret_cast<float4*>(dz + 8 * g);
      float4* t4 = reinterpret_cast<float4*>(tz + 8 * g);
      if (has_draft) {
        d4[0] = make_float4(zs[0], zs[1], zs[2], zs[3]);
        d4[1] = make_float4(zs[4], zs[5], zs[6], zs[7]);
      }
      t4[0] = make_float4(ts[0], ts[1], ts[2], ts[3]);
      t4[1] = make_float4(ts[4], ts[5], ts[6], ts[7]);
    } else {
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int v = 8 * g + j;
        if (v < V) {
          if (has_draft) dz[v] = zs[j];
          tz[v] = ts[j];
        }
      }
    }
  }
  if (!has_draft) return;     // the verifier's extra row has no drafted token
  // block argmax, lowest index among equal maxima
  for (int o = 16; o; o >>= 1) {
    const float ob = __shfl_xor_sync(0xFFFFFFFFu, best, o);
    const int oi = __shfl_xor_sync(0xFFFFFFFFu, bidx, o);
    if (ob > best || (ob == best && oi < bidx)) { best = ob; bidx = oi; }
  }
  __shared__ float sb[kThreads / 32];
  __shared__ int si[kThreads / 32];
  __shared__ float pb[kParts];               // part 0: each part's maximum
  __shared__ int pi[kParts];
  if (lane == 0) { sb[warp] = best; si[warp] = bidx; }
  __syncthreads();
  cg::cluster_group cl = cg::this_cluster();
  if (threadIdx.x == 0) {
    for (int w = 1; w < kThreads / 32; ++w)
      if (sb[w] > best || (sb[w] == best && si[w] < bidx)) { best = sb[w]; bidx = si[w]; }
  }
  cl.sync();                                 // every part has started
  if (threadIdx.x == 0) {
    *cl.map_shared_rank(pb + part, 0) = best;
    *cl.map_shared_rank(pi + part, 0) = bidx;
  }
  cl.sync();
  if (part == 0 && threadIdx.x == 0) {
    for (int p = 1; p < kParts; ++p)
      if (pb[p] > best || (pb[p] == best && pi[p] < bidx)) { best = pb[p]; bidx = pi[p]; }
    tokens[(size_t)b * K_max + i] = bidx;
  }
}

}  // namespace

extern "C" int cmsd_gen_decode_rows(const float* table, const float* heights_it, uint32_t it, int B,
                                    int K_max, int Kt, int V, const int32_t* k_row, uint64_t seed,
                                    float* draft, float* target, int32_t* tokens, void* stream) {
  if (B < 0 || K_max < 1 || V < 2 || (Kt != K_max && Kt != K_max + 1)) return -1;
  if (B == 0) return 0;
  if (!table || !heights_it || !draft || !target || !tokens) return -1;
  const int64_t slots = (int64_t)B * Kt;        // (as many launches as a grid of 2^31 - 1 CTAs needs: one)
  if (slots > 0x7FFFFFFFll) return -1;
  constexpr int kMostSlots = 0x7FFFFFFF / kParts;
  const bool single = (V & 3) != 0 || ((((uintptr_t)draft) | ((uintptr_t)target)) & 15) != 0;
  cudaLaunchConfig_t cfg = {};
  cfg.blockDim = dim3(kThreads);
  cfg.stream = (cudaStream_t)stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  for (int64_t s0 = 0; s0 < slots; s0 += kMostSlots) {
    const int64_t n = slots - s0 < kMostSlots ? slots - s0 : kMostSlots;
    cfg.gridDim = dim3((unsigned)(n * kParts));
    if (cudaLaunchKernelEx(&cfg, single ? gen_rows_kernel<true> : gen_rows_kernel<false>, table, heights_it, it, (int)s0,
                           B, K_max, Kt, V, k_row, cmsd::seed_lo(seed), cmsd::seed_hi(seed), draft, target,
                           tokens) != cudaSuccess)
      return -3;
  }
  return 0;
}
