// Passes over many rows (prefill chunks, serving batches of more than 128 stair rows; up to 128 the GEMMs are mid.cuh's): one launch per
// GEMM and per attention layer, everything a layer needs besides the contractions folded into their
// epilogues.  The persistent kernel streams all weights once per 64 rows, so it is HBM-bound however
// long the prompt is; here a tile holds 128 or 256 rows and the weights are read once per pass.
//
// k_wide_gemm: out[t, n] = sum_k X[t, k] * W[n, k].  The activation rows are the MMA's M side (one TMEM
// lane per row, so everything per row - norm statistics, rotation, argmax - stays in one thread), the
// weight rows its N side.  X is kept as bf16 hi + lo like in the persistent kernel; both parts multiply
// the same weight tile into the same accumulator (hi then lo per 16-element k-step), which makes the
// tensor pipe's work twice the useful work and the loads per MMA smaller than a plain GEMM's.
// CG = 1: 128-row tiles, one CTA each.  CG = 2: 256-row tiles on a CTA pair (cta_group::2): either CTA
// loads its 128 rows of X and half of the weight tile, which takes the shared-memory fill from 64 to 48
// bytes per cycle and SM at 256 columns (measured at the 7B gate/up GEMM, see wide_plan).
//
// Warp roles (352 threads): warps 0 and 10 TMA producers of the weight and the activation tiles (a copy costs its
// issuing thread 200 cycles and more: three copies per k-block from one thread took 0.43 us, the MMAs of a
// 64-column tile 0.22), warp 1 MMA issuer and TMEM owner, warps 2-9 epilogue
// (two per TMEM lane quadrant, alternating chunks).  An accumulator row belongs to one thread, and memory wants
// rows in contiguous pieces, so chunks change hands through a small shared tile per warp.  Two accumulators in TMEM let a tile's epilogue run under the next
// tile's MMAs.  Launches are chained with programmatic dependent launch: a kernel sets itself up and
// fetches its first weight tiles while its predecessor finishes, and touches what the predecessor wrote
// only after griddepcontrol.wait.  All waits are bounded like everywhere in this library.
#pragma once
#include <type_traits>

#include "megakernel.cuh"

namespace stairs {
namespace wide {

using namespace tc;
using mk::store_split4;
using mk::pack_f16x2;
using mk::tma_load_2d_nohint;

constexpr int WM = 128;                    // rows per CTA
constexpr int EPI_WARPS = 8;               // two per TMEM lane quadrant, alternate column chunks
constexpr int WTHREADS = 96 + EPI_WARPS * 32;
constexpr int W_MAX_STAGES = 8;
constexpr int ECH = 16;                    // accumulator columns per epilogue chunk
constexpr int ST_LD = 20;                  // row pitch (floats) of a warp's 32 x 16 exchange tile
constexpr int QT_LD = 36;                  // the same memory as 16 rows x 16 rotation pairs (QKV)
constexpr int ST_BYTES = EPI_WARPS * (32 * ST_LD + 64) * 4;   // (and 64 folded-normalisation constants per warp)

enum WEpi { W_ADD = 0, W_GELU = 1, W_SWIGLU = 2, W_QKV = 3, W_LMHEAD = 4 };

struct WideJob {
  CUtensorMap x_map;        // [2 parts][lo_row rows][K]; box 64 x 128 x 2 (mid.cuh: 64 x x_box x 1)
  CUtensorMap w_map[3];     // box 64 x TN / CG rows; SwiGLU: gate and up matrix, box 64 x TN / 2 rows
  int n_src, src_tiles[3], src_rows[3];
  int src0;                 // W_QKV: first source present (0: q, k, v; 1: k and v only)
  int x_box;                // mid.cuh: rows of the activation box
  int T, TN, n_tiles, m_tiles, kblocks, splits, stages;
  int lo_row;               // rows between the hi and the lo part of every bf16 operand
  int epi;
  int N, ldo;               // output features (SwiGLU: of one matrix), leading dimension of the output
  float* out_f32;           // W_ADD: the residual stream; W_LMHEAD: logits (may be null)
  bf16* out_act;            // W_GELU / W_SWIGLU: ff; W_ADD with next_g: the next operand
  const float* next_g;
  // folded normalisation of the operand (see the persistent kernel)
  int norm_in, norm_kind, d; float eps;
  const float4* stats_in; int stat_tiles_in;    // (mean, M2, count) per row and column tile of x
  float4* stats_out;                            // W_ADD with next_g: [row][2 * n_tiles] (the two warps of a row)
  const float* u; const float* c; int u_off[3], u_last;   // (u_off: first entry of each source, u_last: last entry)
  // W_QKV
  int hd, rope; float qscale;
  const float* rope_cs; const float* rope_sn;   // [row][hd / 2]
  const int* kv_row;                            // cache row of every row's position
  __half* q16; __half* kc; __half* vc;
  unsigned long long* keys;                     // W_LMHEAD
  float* partial; int* counters;                // split tiles
  unsigned int* status; unsigned long long wait_limit;
};

__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <int CG> __device__ __forceinline__ void w_tma(void* dst, const CUtensorMap* map, int c0, int c1, uint64_t* bar, uint64_t policy) {
  if (CG == 1) { tma_load_2d(dst, map, c0, c1, bar, policy); return; }
  // completion is signalled on the pair's even CTA: its copy of the barrier has the same offset
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint"
      " [%0], [%1, {%2, %3}], [%4], %5;"
      ::"r"(smem_u32(dst)), "l"(map), "r"(c0), "r"(c1), "r"(smem_u32(bar) & 0xFEFFFFFFu), "l"(policy) : "memory");
}
template <int CG> __device__ __forceinline__ void w_tma3(void* dst, const CUtensorMap* map, int c0, int c1, int c2, uint64_t* bar, uint64_t policy) {
  if (CG == 1) { mk::tma_load_3d(dst, map, c0, c1, c2, bar, policy); return; }
  asm volatile(
      "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint"
      " [%0], [%1, {%2, %3, %4}], [%5], %6;"
      ::"r"(smem_u32(dst)), "l"(map), "r"(c0), "r"(c1), "r"(c2), "r"(smem_u32(bar) & 0xFEFFFFFFu), "l"(policy) : "memory");
}
template <int CG> __device__ __forceinline__ void w_mma(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
  if (CG == 1) { umma_bf16(d, a, b, idesc, acc); return; }
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d), "l"(a), "l"(b), "r"(idesc), "r"(acc) : "memory");
}
template <int CG> __device__ __forceinline__ void w_commit(uint64_t* bar) {   // CG 2: arrives on both CTAs' copies of the barrier
  if (CG == 1) { umma_commit(bar); return; }
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
               ::"r"(smem_u32(bar)), "h"((uint16_t)3) : "memory");
}
// arrival on the pair leader's copy of a barrier
template <int CG> __device__ __forceinline__ void w_arrive_leader(uint64_t* bar) {
  if (CG == 1) { mbar_arrive(bar); return; }
  uint32_t remote;
  asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(remote) : "r"(smem_u32(bar)));
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(remote) : "memory");
}
template <int CG> __device__ __forceinline__ void w_alloc(uint32_t* slot, uint32_t cols) {
  if (CG == 1) { tmem_alloc(slot, cols); return; }
  asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(slot)), "r"(cols) : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
template <int CG> __device__ __forceinline__ void w_dealloc(uint32_t addr, uint32_t cols) {
  if (CG == 1) { tmem_dealloc(addr, cols); return; }
  asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(addr), "r"(cols) : "memory");
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %cluster_ctarank;" : "=r"(r));
  return r;
}

__device__ __forceinline__ void tmem_ld8(uint32_t taddr, float* v) {
  uint32_t r[8];
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];\n\t"
               "tcgen05.wait::ld.sync.aligned;"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]) : "r"(taddr));
#pragma unroll
  for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(r[i]);
}
__device__ __forceinline__ void tmem_ld16w(uint32_t taddr, float* v) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}
__device__ __forceinline__ void group_sync() { asm volatile("bar.sync 1, 256;" ::: "memory"); }   // the epilogue warps

// packed fp32 arithmetic
__device__ __forceinline__ float2 add2(float2 a, float2 b) {
  float2 r;
  asm("{\n\t.reg .b64 x, y, z;\n\tmov.b64 x, {%2, %3};\n\tmov.b64 y, {%4, %5};\n\tadd.rn.f32x2 z, x, y;\n\tmov.b64 {%0, %1}, z;\n\t}"
      : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return r;
}
__device__ __forceinline__ float2 mul2(float2 a, float2 b) {
  float2 r;
  asm("{\n\t.reg .b64 x, y, z;\n\tmov.b64 x, {%2, %3};\n\tmov.b64 y, {%4, %5};\n\tmul.rn.f32x2 z, x, y;\n\tmov.b64 {%0, %1}, z;\n\t}"
      : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return r;
}
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
  float2 r;
  asm("{\n\t.reg .b64 x, y, w, z;\n\tmov.b64 x, {%2, %3};\n\tmov.b64 y, {%4, %5};\n\tmov.b64 w, {%6, %7};\n\tfma.rn.f32x2 z, x, y, w;\n\tmov.b64 {%0, %1}, z;\n\t}"
      : "=f"(r.x), "=f"(r.y) : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
  return r;
}

// GELU(v) = v / 2 * erfc(-v / sqrt 2).  Within |v| < 1: 1 + erf(v / sqrt 2) by a polynomial; outside, with z = |v| / sqrt 2 and
// t = 1 / (1 + 0.4 z), erfc(z) = t P(t) exp(-z^2), which does not cancel for negative v.  Both polynomials are minimax fits (Remez
// exchange) of erf(v / sqrt 2) / v in v^2, relative error 7e-10, and of exp(z^2) erfc(z) / t in t for z of 0.707 to 9.9, 1e-7.
// Largest relative error against 64 bits on the device (of the erff form): v in [-1, 1) 2.6e-7 (2.1e-7), [1, 13) 1.5e-7 (1.2e-7),
// [-2, -1) 6e-7 (1.2e-6), [-4, -2) 9e-7 (9e-4), [-8, -4) 2.8e-6 (1); root mean square at most the erff form's but for [-1, -0.5), 6.6e-8
// (6.0e-8).  The result is kept to 7.6e-6 (bf16 hi + lo).
// The epilogue warps' issue rate bounds the GEMM (0.4B fc1 over 2048 rows; erff has twice the instructions): two values at a
// time, packed fp32 arithmetic halves what the polynomials issue.
__device__ __forceinline__ float2 gelu_erfc2(float2 v) {
  auto k2 = [](float k) { return make_float2(k, k); };
  const float2 s = mul2(v, v), d = fma2(make_float2(fabsf(v.x), fabsf(v.y)), k2(0.28284271247461901f), k2(1.0f));
  const float2 t = make_float2(__fdividef(1.0f, d.x), __fdividef(1.0f, d.y)), x = mul2(s, k2(-0.72134752044448170f));   // exp(-z^2) = 2^(-s / (2 ln 2))
  float2 p = fma2(t, k2(-0.11336128f), k2(0.23559201f));
  p = fma2(t, p, k2(0.017188916f)); p = fma2(t, p, k2(0.2079364f)); p = fma2(t, p, k2(0.20036721f)); p = fma2(t, p, k2(0.2264413f)); p = fma2(t, p, k2(0.22564292f));
  const float2 c = mul2(mul2(t, p), make_float2(mk::fast_exp2(x.x), mk::fast_exp2(x.y)));   // erfc(z)
  float2 q = fma2(s, k2(-1.53084166e-5f), k2(2.26972741e-4f));
  q = fma2(s, q, k2(-2.37265998e-3f)); q = fma2(s, q, k2(1.99466459e-2f)); q = fma2(s, q, k2(-0.132980719f)); q = fma2(s, q, k2(0.797884583f));
  q = fma2(v, q, k2(1.0f));
  const float2 r = make_float2(s.x < 1.0f ? q.x : v.x < 0.f ? c.x : 2.0f - c.x, s.y < 1.0f ? q.y : v.y < 0.f ? c.y : 2.0f - c.y);
  return mul2(mul2(v, k2(0.5f)), r);
}

// TMEM columns of two accumulators of TN columns (an allocation is a power of two of at least 32); the second one starts halfway
__host__ __device__ inline int tmem_columns(int TN) {
  int c = 32;
  while (c < 2 * TN) c <<= 1;
  return c;
}

// ---------------------------------------------------------------------------------------------
// The GEMM
// ---------------------------------------------------------------------------------------------
template <int CG>
__global__ void __launch_bounds__(WTHREADS, 1) k_wide_gemm(const __grid_constant__ WideJob job) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  const int TN = job.TN, TNc = TN / CG, stages = job.stages, S = job.splits;
  constexpr int a_bytes = WM * BK * 2;                               // one part of the activation tile
  const int stage_bytes = 2 * a_bytes + TNc * BK * 2;
  uint8_t* tail = smem + (size_t)stages * stage_bytes;
  float* stile = reinterpret_cast<float*>(tail);                     // [EPI_WARPS][32][ST_LD]
  uint64_t* full = reinterpret_cast<uint64_t*>(tail + ST_BYTES);
  uint64_t* empty = full + W_MAX_STAGES;
  uint64_t* acc_full = empty + W_MAX_STAGES;                         // [2]
  uint64_t* acc_empty = acc_full + 2;                                // [2]
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_empty + 2);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  volatile int* verdict = abort_flag + 1;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = CG == 2 ? (int)cluster_rank() : 0;
  const int cid = blockIdx.x / CG, G = gridDim.x / CG;               // this CTA (pair) among the CTAs (pairs)
  const int units = job.n_tiles * job.m_tiles * S;                   // one unit: a K range of one tile
  const uint32_t tmem_cols = tmem_columns(TN);

  if (threadIdx.x == 0) {
    for (int s = 0; s < stages; ++s) { mbar_init(full + s, 1); mbar_init(empty + s, 1); }
    mbar_init(acc_full + 0, 1); mbar_init(acc_full + 1, 1);
    mbar_init(acc_empty + 0, EPI_WARPS * CG); mbar_init(acc_empty + 1, EPI_WARPS * CG);
    *abort_flag = 0; *verdict = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) w_alloc<CG>(tmem_slot, tmem_cols);
  tc_fence_before();
  if (CG == 2) cluster_sync(); else __syncthreads();
  tc_fence_after();
  if (CG == 2) __syncthreads();
  const uint32_t tmem_base = *tmem_slot;
  if (threadIdx.x == 0) pdl_launch();   // (after the TMEM allocation, see k_wide_attn_tc)
  int issued = 0, p_stage = 0;
  uint32_t p_phase = 0;
  auto k_begin = [&](int s) { return (job.kblocks * s) / S; };

  if (warp == 0) {
    // ------------------------------------------------------------------ TMA producer, weight tiles
    // (they depend on nothing: fetched while the predecessor still runs)
    if (lane == 0) {
      const uint64_t pol_w = policy_evict_first();
      const uint32_t tx = (uint32_t)(CG * stage_bytes);   // both parts, both CTAs
      int stage = 0; uint32_t phase = 0;
      bool ok = true;
      for (int u = cid; u < units && ok; u += G) {
        const int s = u % S, nt = (u / S) / job.m_tiles;
        int src = 0, local = nt;
        while (src + 1 < job.n_src && local >= job.src_tiles[src]) { local -= job.src_tiles[src]; ++src; }
        // SwiGLU tile: TN / 2 gate rows and the same up rows (either CTA of a pair holds one of them)
        const bool glu = job.epi == W_SWIGLU;
        const int row = glu ? local * (TN / 2) : local * TN + rank * TNc;
        const CUtensorMap* map = &job.w_map[glu ? rank : src];
        const int kb0 = k_begin(s), len = k_begin(s + 1) - kb0;
        for (int kb = kb0; kb < kb0 + len; ++kb) {
          if (!mbar_wait(empty + stage, phase ^ 1, abort_flag, job.wait_limit)) { ok = false; break; }
          uint8_t* dst = smem + (size_t)stage * stage_bytes + 2 * a_bytes;
          if (rank == 0) mbar_expect_tx(full + stage, tx);
          w_tma<CG>(dst, map, kb * BK, row, full + stage, pol_w);
          if (glu && CG == 1) w_tma<CG>(dst + (TN / 2) * BK * 2, &job.w_map[1], kb * BK, row, full + stage, pol_w);
          ++issued;
          if (++stage == stages) { stage = 0; phase ^= 1; }
          p_stage = stage; p_phase = phase;
        }
      }
    }
  } else if (warp == 10) {
    // ------------------------------------------------------------------ TMA producer, activation tiles
    if (lane == 0) {
      const uint64_t pol_x = policy_evict_last();
      pdl_wait();
      int stage = 0; uint32_t phase = 0;
      bool ok = true;
      for (int u = cid; u < units && ok; u += G) {
        const int s = u % S, mt = (u / S) % job.m_tiles;
        const int x_row = (mt * CG + rank) * WM;
        const int kb0 = k_begin(s), len = k_begin(s + 1) - kb0;
        for (int kb = kb0; kb < kb0 + len; ++kb) {
          if (!mbar_wait(empty + stage, phase ^ 1, abort_flag, job.wait_limit)) { ok = false; break; }
          w_tma3<CG>(smem + (size_t)stage * stage_bytes, &job.x_map, kb * BK, x_row, 0, full + stage, pol_x);   // hi rows, then lo rows
          if (++stage == stages) { stage = 0; phase ^= 1; }
        }
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer (the pair's even CTA)
    if (lane == 0 && rank == 0) {
      // fp32 accumulator, bf16 operands, both K-major, M = 128 * CG, N = TN
      const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(TN >> 3) << 17) | ((uint32_t)((WM * CG) >> 4) << 24);
      int stage = 0; uint32_t phase = 0;
      int buf = 0; uint32_t acc_bits = 0;
      bool ok = true;
      for (int u = cid; u < units && ok; u += G) {
        const int s = u % S;
        if (!mbar_wait(acc_empty + buf, ((acc_bits >> buf) & 1u) ^ 1u, abort_flag, job.wait_limit)) break;
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + (uint32_t)buf * (tmem_cols / 2);
        const int kb0 = k_begin(s), kb1 = k_begin(s + 1);
        for (int kb = kb0; kb < kb1; ++kb) {
          if (!mbar_wait(full + stage, phase, abort_flag, job.wait_limit)) { ok = false; break; }
          tc_fence_after();
          const uint32_t a = smem_u32(smem + (size_t)stage * stage_bytes);
          const uint64_t hi = smem_desc_sw128(a), lo = smem_desc_sw128(a + a_bytes), w = smem_desc_sw128(a + 2 * a_bytes);
#pragma unroll
          for (int k = 0; k < BK / UMMA_K; ++k) {
            const uint64_t o = (uint64_t)(k * UMMA_K * 2 / 16);
            w_mma<CG>(d_tmem, hi + o, w + o, idesc, (kb > kb0 || k > 0) ? 1u : 0u);
            w_mma<CG>(d_tmem, lo + o, w + o, idesc, 1u);
          }
          w_commit<CG>(empty + stage);
          if (++stage == stages) { stage = 0; phase ^= 1; }
        }
        if (!ok) break;
        w_commit<CG>(acc_full + buf);
        acc_bits ^= 1u << buf; buf ^= 1;
      }
    }
  } else {
    // ------------------------------------------------------------------ epilogue (warps 2..9)
    const int quad = warp & 3, hw = (warp - 2) >> 2, et = threadIdx.x - 64;
    float* st = stile + (size_t)(warp - 2) * (32 * ST_LD + 64);
    float* uc = st + 32 * ST_LD;
    const int tr = lane >> 2, tc4 = (lane & 3) * 4;    // exchange-tile mapping: row 8 i + tr, four columns from tc4
    int buf = 0; uint32_t acc_bits = 0;
    pdl_wait();
    for (int u = cid; u < units; u += G) {
      const int sp = u % S, tile = u / S, nt = tile / job.m_tiles, mt = tile % job.m_tiles;
      const int row0 = (mt * CG + rank) * WM + quad * 32, row = row0 + lane;
      const bool row_on = row < job.T;
      int src = 0, local = nt;
      while (src + 1 < job.n_src && local >= job.src_tiles[src]) { local -= job.src_tiles[src]; ++src; }
      const int col0 = local * TN;                      // first weight row of the tile in its source
      // What the epilogue reads from memory is requested before the accumulator is waited for, and inside
      // the loops a few chunks ahead: every such load is an L2 round trip.
      float rs = 1.f, mu = 0.f;
      if (job.norm_in && row_on) {
        // one pass over the row's tile entries, eight loads in flight; sums shifted by the first tile's mean
        const float4* sr = job.stats_in + (size_t)row * job.stat_tiles_in;
        float n = 0.f, s1 = 0.f, s2 = 0.f, m0 = 0.f;
        for (int i0 = 0; i0 < job.stat_tiles_in; i0 += 8) {
          float4 e[8];
#pragma unroll
          for (int i = 0; i < 8; ++i) e[i] = i0 + i < job.stat_tiles_in ? __ldcg(sr + i0 + i) : make_float4(0.f, 0.f, 0.f, 0.f);
          if (i0 == 0) m0 = e[0].x;
#pragma unroll
          for (int i = 0; i < 8; ++i) { const float d0 = e[i].x - m0, nd = e[i].z * d0; n += e[i].z; s1 += nd; s2 += e[i].y + nd * d0; }
        }
        const float dm = s1 / fmaxf(n, 1.f), mean = m0 + dm, m2 = fmaxf(s2 - s1 * dm, 0.f);
        if (job.norm_kind == 0) { mu = mean; rs = 1.0f / sqrtf(m2 / (float)job.d + job.eps); }
        else rs = 1.0f / sqrtf((m2 + n * mean * mean) / (float)job.d + job.eps);
      }
      // this warp's chunk i covers tile columns col_of(i) .. col_of(i) + 15
      auto col_of = [&](int i) { return (2 * i + hw) * ECH; };
      // old residual values of the chunk at c0; four chunks are kept in flight
      float4 xq[4][4];                                  // (QKV: rotation table entries in xq[0], xq[1], see load_rope)
      auto load_x = [&](float4 (&q)[4], int c0) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int r = row0 + 8 * i + tr;
          q[i] = (r < job.T && c0 < TN && col0 + c0 < job.N) ? __ldcg(reinterpret_cast<const float4*>(job.out_f32 + (size_t)r * job.ldo + col0 + c0 + tc4))
                                                             : make_float4(0.f, 0.f, 0.f, 0.f);
        }
      };
      auto load_x_first = [&]() {
#pragma unroll
        for (int j = 0; j < 4; ++j) load_x(xq[j], col_of(j));
      };
      if (job.epi == W_ADD && S == 1) load_x_first();
      // QKV: item `it` holds 16 rotation pairs of a head (columns i0 .. i0 + 15 and half a head further); in the
      // exchange tile four lanes hold a row's pairs, rows 8 i + (lane >> 2) of a half chunk
      const int part = src + job.src0, half = job.hd / 2, gph = job.epi == W_QKV ? (half + 15) / 16 : 1;
      const bool rot = job.epi == W_QKV && job.rope && part < 2;
      auto load_rope = [&](float4 (&q)[4], int it, int h) {   // cos and sin of the two rows of half chunk h
        const int i0 = (it % gph) * 16 + tc4;
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const int r = row0 + 16 * h + 8 * i + tr;
          const size_t o = (size_t)(r < job.T ? r : 0) * half + (i0 < half ? i0 : 0);
          q[2 * i] = __ldcg(reinterpret_cast<const float4*>(job.rope_cs + o));
          q[2 * i + 1] = __ldcg(reinterpret_cast<const float4*>(job.rope_sn + o));
        }
      };
      int kv_row[4];                                    // cache rows of this lane's rows (two per half chunk)
      if (job.epi == W_QKV) {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int r = row0 + 8 * j + tr;
          kv_row[j] = part == 0 ? r : (r < job.T ? __ldcg(job.kv_row + r) : 0);
        }
        if (rot) {
#pragma unroll
          for (int j = 0; j < 2; ++j) load_rope(xq[j], hw, j);
        }
      }
      bool ok = mbar_wait(acc_full + buf, (acc_bits >> buf) & 1u, abort_flag, job.wait_limit);
      ok = __all_sync(0xffffffffu, ok);
      if (S > 1) {   // the split tiles' barriers below want one verdict for the whole group
        if (!ok) *abort_flag = 1;
        group_sync();
        if (et == 0) *verdict = *abort_flag ? 0 : 1;
        group_sync();
        ok = *verdict != 0;
      }
      if (!ok) break;
      acc_bits ^= 1u << buf;
      tc_fence_after();
      const uint32_t taddr = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)buf * (tmem_cols / 2);
      bool finish = true;
      const size_t part_stride = (size_t)TN * WM;
      const float* parts = job.partial + (size_t)tile * S * part_stride + (size_t)(quad * 32 + lane) * 4;
      if (S > 1) {
        // a K range of the tile: park it ([4 columns][row] vectors), the last arriver adds the ranges in K order
        float* mine = const_cast<float*>(parts) + (size_t)sp * part_stride;
        for (int c0 = hw * 8; c0 < TN; c0 += 16) {
          float v[8];
          tmem_ld8(taddr + (uint32_t)c0, v);
          if (row_on) {
            *reinterpret_cast<float4*>(mine + (size_t)c0 * WM) = make_float4(v[0], v[1], v[2], v[3]);
            *reinterpret_cast<float4*>(mine + (size_t)(c0 + 4) * WM) = make_float4(v[4], v[5], v[6], v[7]);
          }
        }
        __threadfence();
        group_sync();
        if (et == 0) {
          const int old = atomicAdd(job.counters + tile, 1);
          if (old == S - 1) job.counters[tile] = 0;
          *verdict = old == S - 1 ? 2 : 1;
        }
        group_sync();
        finish = *verdict == 2;
        if (finish) {
          __threadfence();
          if (job.epi == W_ADD) load_x_first();
        }
      }
      // 16 consecutive accumulator columns of this thread's row
      auto acc = [&](int c0, float* v) {
        constexpr int NC = 16;
        if (S == 1) {
          tmem_ld16w(taddr + (uint32_t)c0, v);
          return;
        }
#pragma unroll
        for (int j = 0; j < NC; ++j) v[j] = 0.f;
        if (row_on) {
          const float* p0 = parts + (size_t)c0 * WM;
#pragma unroll 4
          for (int s2 = 0; s2 < S; ++s2) {
            float4 a[NC / 4];
#pragma unroll
            for (int j = 0; j < NC / 4; ++j) a[j] = __ldcg(reinterpret_cast<const float4*>(p0 + s2 * part_stride + (size_t)(4 * j) * WM));
#pragma unroll
            for (int j = 0; j < NC / 4; ++j) { v[4 * j] += a[j].x; v[4 * j + 1] += a[j].y; v[4 * j + 2] += a[j].z; v[4 * j + 3] += a[j].w; }
          }
        }
      };
      // Folded normalisation of 16 columns.  Their constants u and c (LayerNorm models) are fetched a chunk ahead,
      // one per lane, and handed out through shared memory: read per column they were two dependent
      // round trips in every chunk (0.4B fc1 over 2048 rows: 54 -> 45 us).
      auto fetch_uc = [&](int n) { return job.u ? __ldg((lane < 16 ? job.u : job.c) + min(n + (lane & 15), job.u_last)) : 0.f; };
      auto share_uc = [&](float a, float b) {
        if (job.u) { __syncwarp(); uc[lane] = a; uc[32 + lane] = b; __syncwarp(); }
      };
      auto normed = [&](float* v, int group) {
        if (!job.u) {
#pragma unroll
          for (int j = 0; j < 16; ++j) v[j] *= rs;
          return;
        }
#pragma unroll
        for (int j = 0; j < 16; j += 4) {
          const float4 u4 = *reinterpret_cast<const float4*>(uc + 32 * group + j), c4 = *reinterpret_cast<const float4*>(uc + 32 * group + 16 + j);
          v[j] = rs * (v[j] - mu * u4.x) + c4.x; v[j + 1] = rs * (v[j + 1] - mu * u4.y) + c4.y;
          v[j + 2] = rs * (v[j + 2] - mu * u4.z) + c4.z; v[j + 3] = rs * (v[j + 3] - mu * u4.w) + c4.w;
        }
      };
      auto to_tile = [&](const float* v) {
        __syncwarp();
#pragma unroll
        for (int j = 0; j < 4; ++j) *reinterpret_cast<float4*>(st + lane * ST_LD + 4 * j) = make_float4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
        __syncwarp();
      };
      auto store_act = [&](int out_col) {   // the exchange tile as bf16 hi + lo, a 32-byte sector per row and part
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int r = row0 + 8 * i + tr;
          if (r < job.T)
            store_split4(job.out_act, (size_t)r * job.ldo + out_col + tc4, (size_t)job.lo_row * job.ldo, *reinterpret_cast<const float4*>(st + (8 * i + tr) * ST_LD + tc4));
        }
      };
      if (finish) {
        if (job.epi == W_ADD) {
          // residual update, the next GEMM's operand bf16(x * gain), and this warp's row statistics of the tile: mean and centred sum of
          // squares of four values a lane and chunk, merged pair by pair (Chan, Golub and LeVeque's formula).  Sums shifted by one of the
          // row's values, in one pass, lose up to seven bits where that value is an outlier channel's.
          float mean[4], m2[4];
#pragma unroll
          for (int i = 0; i < 4; ++i) mean[i] = m2[i] = 0.f;
          const int nch = (min(TN, job.N - col0) / ECH - hw + 1) / 2;   // this warp's chunks
          for (int k0 = 0; k0 < nch; k0 += 4) {
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              if (k0 + j < nch) {
                const int c0 = col_of(k0 + j), col = col0 + c0 + tc4;
                float v[16];
                acc(c0, v);
                to_tile(v);
                const float4 g4 = job.next_g ? __ldg(reinterpret_cast<const float4*>(job.next_g + col)) : make_float4(0.f, 0.f, 0.f, 0.f);
                const float share = 1.0f / (float)(k0 + j + 1), weight = 4.0f * (float)(k0 + j) * share;   // (4 values after 4 (k0 + j))
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                  const int r = row0 + 8 * i + tr;
                  const float4 a = *reinterpret_cast<const float4*>(st + (8 * i + tr) * ST_LD + tc4);
                  const float4 x4 = make_float4(xq[j][i].x + a.x, xq[j][i].y + a.y, xq[j][i].z + a.z, xq[j][i].w + a.w);
                  if (r < job.T) {
                    *reinterpret_cast<float4*>(job.out_f32 + (size_t)r * job.ldo + col) = x4;
                    if (job.next_g)
                      store_split4(job.out_act, (size_t)r * job.ldo + col, (size_t)job.lo_row * job.ldo, make_float4(x4.x * g4.x, x4.y * g4.y, x4.z * g4.z, x4.w * g4.w));
                  }
                  const float m = 0.25f * ((x4.x + x4.y) + (x4.z + x4.w)), dm = m - mean[i];
                  const float d0 = x4.x - m, d1 = x4.y - m, d2 = x4.z - m, d3 = x4.w - m;
                  m2[i] += ((d0 * d0 + d1 * d1) + (d2 * d2 + d3 * d3)) + dm * dm * weight;
                  mean[i] += dm * share;
                }
                load_x(xq[j], col_of(k0 + j + 4));
              }
            }
          }
          if (job.next_g) {
            const float cnt = (float)(nch * ECH);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
#pragma unroll
              for (int o = 1; o < 4; o <<= 1) {   // (as many values on either side: cnt / 4, then cnt / 2)
                const float m = __shfl_xor_sync(0xffffffffu, mean[i], o), q = __shfl_xor_sync(0xffffffffu, m2[i], o), dm = m - mean[i];
                m2[i] = (m2[i] + q) + dm * dm * (0.125f * (float)o * cnt);
                mean[i] = 0.5f * (mean[i] + m);
              }
              const int r = row0 + 8 * i + tr;
              if ((lane & 3) == 0 && r < job.T) job.stats_out[(size_t)r * (2 * job.n_tiles) + 2 * nt + hw] = make_float4(mean[i], m2[i], cnt, 0.f);
            }
          }
        } else if (job.epi == W_GELU) {
          float ua = fetch_uc(col0 + col_of(0));
          for (int i = 0; col_of(i) < TN && col0 + col_of(i) < job.N; ++i) {
            const int n = col0 + col_of(i);
            float v[16];
            share_uc(ua, 0.f);
            ua = fetch_uc(col0 + col_of(i + 1));
            acc(col_of(i), v);
            normed(v, 0);
#pragma unroll
            for (int j = 0; j < 16; j += 2) { const float2 g2 = gelu_erfc2(make_float2(v[j], v[j + 1])); v[j] = g2.x; v[j + 1] = g2.y; }
            to_tile(v);
            store_act(n);
          }
        } else if (job.epi == W_SWIGLU) {
          const int out0 = local * (TN / 2);             // output columns of the tile
          float ua = fetch_uc(out0 + col_of(0)), ub = fetch_uc(job.N + out0 + col_of(0));
          for (int i = 0; col_of(i) < TN / 2; ++i) {
            const int oc = col_of(i), n = out0 + oc;
            if (n >= job.N) break;
            float v[16], w[16];
            share_uc(ua, ub);
            ua = fetch_uc(out0 + col_of(i + 1)); ub = fetch_uc(job.N + out0 + col_of(i + 1));
            acc(oc, v);
            acc(oc + TN / 2, w);
            normed(v, 0);
            normed(w, 1);
#pragma unroll
            for (int j = 0; j < 16; ++j) v[j] = silu_f(v[j]) * w[j];
            to_tile(v);
            store_act(n);
          }
        } else if (job.epi == W_LMHEAD) {
          unsigned long long key = 0ull;
          float ua = fetch_uc(col0 + col_of(0));
          for (int i = 0; col_of(i) < TN && col0 + col_of(i) < job.N; ++i) {
            const int n0 = col0 + col_of(i);
            float v[16];
            share_uc(ua, 0.f);
            ua = fetch_uc(col0 + col_of(i + 1));
            acc(col_of(i), v);
            normed(v, 0);
#pragma unroll
            for (int j = 0; j < 16; ++j) {
              const unsigned long long k2 = argmax_key(v[j], (uint32_t)(n0 + j));
              if (n0 + j < job.N && k2 > key) key = k2;
            }
            if (job.out_f32) {
              to_tile(v);
              const int n = n0 + (lane & 15);
              for (int r = lane >> 4; r < 32 && row0 + r < job.T; r += 2)
                if (n < job.N) job.out_f32[(size_t)(row0 + r) * job.ldo + n] = st[r * ST_LD + (lane & 15)];
            }
          }
          if (row_on && key) atomicMax(job.keys + row, key);
        } else {   // W_QKV: rotate and scale q, rotate k; fp16 to the query buffer and the cache
          const int width = job.src_rows[src], u0 = job.u_off[src] + col0;
          __half* dst0 = (part == 0 ? job.q16 : part == 1 ? job.kc : job.vc) + col0;
          const float qs = part == 0 ? job.qscale : 1.0f;
          const int n_it = min(TN, width - col0) / job.hd * gph;
          const int cf = hw / gph * job.hd + (hw % gph) * 16;
          float ua = fetch_uc(u0 + cf), ub = fetch_uc(u0 + cf + half);
          for (int it = hw; it < n_it; it += 2) {
            const int i0 = (it % gph) * 16, c_lo = it / gph * job.hd + i0, c_hi = c_lo + half;
            float v[32];
            share_uc(ua, ub);
            { const int i1 = ((it + 2) % gph) * 16, c1 = (it + 2) / gph * job.hd + i1; ua = fetch_uc(u0 + c1); ub = fetch_uc(u0 + c1 + half); }
            acc(c_lo, v);
            acc(c_hi, v + 16);
            normed(v, 0);
            normed(v + 16, 1);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              __syncwarp();
              if ((lane >> 4) == h) {   // rows 16 h .. 16 h + 15
#pragma unroll
                for (int e = 0; e < 8; ++e) *reinterpret_cast<float4*>(st + (lane & 15) * QT_LD + 4 * e) = make_float4(v[4 * e], v[4 * e + 1], v[4 * e + 2], v[4 * e + 3]);
              }
              __syncwarp();
#pragma unroll
              for (int i = 0; i < 2; ++i) {
                const int rl = 8 * i + tr, r = row0 + 16 * h + rl;
                float4 lo = *reinterpret_cast<const float4*>(st + rl * QT_LD + tc4), hi = *reinterpret_cast<const float4*>(st + rl * QT_LD + 16 + tc4);
                if (rot) {
                  const float4 cs = xq[h][2 * i], sn = xq[h][2 * i + 1], l = lo, g = hi;
                  lo = make_float4(l.x * cs.x - g.x * sn.x, l.y * cs.y - g.y * sn.y, l.z * cs.z - g.z * sn.z, l.w * cs.w - g.w * sn.w);
                  hi = make_float4(g.x * cs.x + l.x * sn.x, g.y * cs.y + l.y * sn.y, g.z * cs.z + l.z * sn.z, g.w * cs.w + l.w * sn.w);
                }
                if (r < job.T && i0 + tc4 < half) {
                  __half* dst = dst0 + (size_t)kv_row[2 * h + i] * width + tc4;
                  *reinterpret_cast<uint2*>(dst + c_lo) = make_uint2(pack_f16x2(lo.x * qs, lo.y * qs), pack_f16x2(lo.z * qs, lo.w * qs));
                  *reinterpret_cast<uint2*>(dst + c_hi) = make_uint2(pack_f16x2(hi.x * qs, hi.y * qs), pack_f16x2(hi.z * qs, hi.w * qs));
                }
              }
              if (rot) load_rope(xq[h], it + 2, h);
            }
          }
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) w_arrive_leader<CG>(acc_empty + buf);
      buf ^= 1;
    }
  }

  // ------------------------------------------------------------------ teardown
  tc_fence_before();
  __syncthreads();
  if (*abort_flag) {
    if (threadIdx.x == 0) {
      *reinterpret_cast<volatile unsigned int*>(job.status + STATUS_ERROR) = 5u;  // STAIRS_ETIMEOUT
      __threadfence_system();
      // copies in flight must land before the shared memory is given back (bounded).  A pair's copies all
      // signal on the even CTA, so the odd one waits out the bound.
      const long long t0 = clock64();
      const unsigned long long lim = job.wait_limit > 2000000ull ? job.wait_limit : 2000000ull;
      int s = p_stage; uint32_t ph = p_phase;
      for (int i = 0; i < stages && i < issued; ++i) {
        if (--s < 0) { s = stages - 1; ph ^= 1; }
        while (rank != 0 || !mbar_try(full + s, ph)) {
          if ((unsigned long long)(clock64() - t0) > lim) break;
        }
      }
      settle(t0);
    }
    __syncthreads();
  }
  if (CG == 2) cluster_sync();   // neither CTA leaves while the other may still use its shared memory or barriers
  if (warp == 1) { tc_fence_after(); w_dealloc<CG>(tmem_base, tmem_cols); }
}

inline size_t gemm_smem(int TN, int CG, int stages) {
  const size_t stage = 2 * (size_t)WM * BK * 2 + (size_t)(TN / CG) * BK * 2;
  return 1024 + stages * stage + ST_BYTES + (2 * W_MAX_STAGES + 4) * 8 + 64;
}
inline int gemm_stages(int TN, int CG) {
  int s = W_MAX_STAGES;
  while (s > 2 && gemm_smem(TN, CG, s) > (size_t)SMEM_LIMIT) --s;
  return s;
}

// ---------------------------------------------------------------------------------------------
// Attention over the paged cache
// ---------------------------------------------------------------------------------------------
struct WideAttn {
  const __half* q16;             // [row][Hq * hd], rotated, scaled by log2(e) / sqrt(hd)
  const __half* kc; const __half* vc;
  bf16* o; int lo_row;           // [row][Hq * hd] hi, lo lo_row rows further down
  const int* page_table; int page_tokens, max_pages;
  // requests: device arrays (slot, draft length, first row), or one prefill chunk when val_req is null
  const int* val_req; const int* val_k; const int* val_off; const int* n_seq;
  int n_qblk;                    // query blocks per request of the launch (blocks past a request's own count leave)
  int slot, first, rows;         // prefill: slot, first position, rows
  int Hq, Hkv, hd;
};

__device__ __forceinline__ uint32_t map_rank(uint32_t addr, uint32_t r) {
  uint32_t o;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(o) : "r"(addr), "r"(r));
  return o;
}
__device__ __forceinline__ float4 ld_cluster_f4(uint32_t addr) {
  float4 v;
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr) : "memory");
  return v;
}

__device__ __forceinline__ float ld_cluster_f1(uint32_t addr) {
  float v;
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(addr) : "memory");
  return v;
}

constexpr int WCH = 64;          // positions per chunk
template <int NW, int MT> constexpr int attn_state_rows() { return (NW / MT) * MT * 16; }
inline size_t attn_smem(int hd, int nw, int mt) {
  const size_t pitch = (size_t)hd * 2 + 16, ring = 4 * WCH * pitch;
  const size_t states = (size_t)nw * 16 * (hd + 4) * 4;
  return std::max(ring, states) + 3 * WCH * 4 + 16;
}

// One block: MT blocks of 16 queries (query q of a request = row q / G, head q % G of the kv head) times
// NW / MT position slices of every 64-position chunk, one warp each, on mma.sync m16n8k16 with the online
// softmax in registers (base 2).  <8, 8> serves prefill chunks (128 queries share a chunk's copies);
// <4, 1..4> requests with few query rows, whose warps split the positions instead, three or four blocks to an SM (16 requests x 32
// heads of 80 are 512 blocks: with 141 registers a thread, three to an SM, the last 68 were a second wave; with 128, 3.5 us less a layer).  Long contexts of few
// blocks are cut over a cluster of up to 8 CTAs (grid z); slices and ranges are merged at the end through
// (distributed) shared memory in a fixed order.  Chunks are staged by 16-byte asynchronous copies, the
// next one under the current one's MMAs.
// EXACT: hd == 16 * KS (loops without guards).
template <int KS, bool EXACT, int NW, int MT>
__global__ void __launch_bounds__(NW * 32, NW == 8 ? (KS <= 5 ? 2 : 1) : (KS <= 5 ? 4 : 3)) k_wide_attn(const __grid_constant__ WideAttn P) {
  extern __shared__ __align__(16) uint8_t asm_raw[];
  constexpr int NP = NW / MT, SL = WCH / NP;       // position slices, positions per slice
  constexpr int RND = SL < 32 ? SL : 32;           // positions per softmax round
  constexpr int NT = RND / 8;
  constexpr int NTH = NW * 32;
  const int hd = P.hd, ksteps = hd / 16, ntiles = hd / 8, G = P.Hq / P.Hkv;
  const int pitch = hd * 2 + 16, kvb = WCH * pitch;
  int* rowbuf = reinterpret_cast<int*>(asm_raw + max((size_t)4 * kvb, (size_t)NW * 16 * (hd + 4) * 4));   // [3][WCH]
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, g = lane >> 2, t4 = lane & 3;
  const int NS = gridDim.z, zr = blockIdx.z;
  if (tid == 0) pdl_launch();
  // (requests, page table and cached positions are older than this pass: read, and the first chunks' copies started, while the
  // predecessor still runs; the queries and this call's own positions are its work)
  int slot, base, R, off;
  const int i_req = blockIdx.y / P.n_qblk, kvh = blockIdx.x;
  int qblk = blockIdx.y % P.n_qblk;
  if (P.val_req) {
    slot = P.val_req[i_req]; R = P.val_k[i_req] + 1; off = P.val_off[i_req]; base = P.n_seq[slot] - 1;
  } else { slot = P.slot; R = P.rows; off = 0; base = P.first; qblk = P.n_qblk - 1 - qblk; }   // (the longest blocks first)
  const int Q = R * G, q0 = qblk * MT * 16;
  if (q0 >= Q) { pdl_wait(); return; }              // (uniform over the cluster)
  const int mt = w % MT, part = w / MT;
  const int nQ = min(MT * 16, Q - q0);
  const int last_pos = base + (q0 + nQ - 1) / G;    // last position any query of the block sees
  const int n_chunks = last_pos / WCH + 1;
  const int c_begin = (n_chunks * zr) / NS, c_end = (n_chunks * (zr + 1)) / NS;
  const int nq = P.Hq * hd, nkv = P.Hkv * hd;
  const int* pt = P.page_table + (size_t)slot * P.max_pages;

  auto look_up = [&](int c) {                       // cache rows of chunk c's positions (-1 past the end)
    if (tid < WCH) {
      const int pz = c * WCH + tid;
      rowbuf[(c % 3) * WCH + tid] = pz <= last_pos ? pt[pz / P.page_tokens] * P.page_tokens + pz % P.page_tokens : -1;
    }
  };
  const int pieces = hd / 8;
  auto stage = [&](int c, int b) {
    uint8_t* kd = asm_raw + (size_t)b * 2 * kvb;
    uint8_t* vd = kd + kvb;
    const int* rows = rowbuf + (c % 3) * WCH;
    int j = tid / pieces, pc = tid % pieces;
    const int dj = NTH / pieces, dp = NTH % pieces;
    while (j < WCH) {
      const int rb = rows[j];
      const size_t src = (size_t)max(rb, 0) * nkv + (size_t)kvh * hd + pc * 8;
      mk::cp_async16(kd + j * pitch + pc * 16, P.kc + src, rb >= 0);
      mk::cp_async16(vd + j * pitch + pc * 16, P.vc + src, rb >= 0);
      j += dj; pc += dp;
      if (pc >= pieces) { pc -= pieces; ++j; }
    }
    mk::cp_async_commit();
  };

  const int ql_a = mt * 16 + g, ql_b = ql_a + 8;
  const bool on_a = ql_a < nQ, on_b = ql_b < nQ;
  const int qa = q0 + (on_a ? ql_a : 0), qb = q0 + (on_b ? ql_b : 0);
  const int last_a = on_a ? base + qa / G : -1, last_b = on_b ? base + qb / G : -1;
  const int warp_first = base + (q0 + mt * 16) / G;                                       // first query's last visible position
  const int warp_last = mt * 16 < nQ ? base + (q0 + min(mt * 16 + 15, nQ - 1)) / G : -1;  // (-1: no queries)
  float m_a = -INFINITY, m_b = -INFINITY, l_a = 0.f, l_b = 0.f;
  float o[2 * KS][4];
#pragma unroll
  for (int nd = 0; nd < 2 * KS; ++nd) o[nd][0] = o[nd][1] = o[nd][2] = o[nd][3] = 0.f;

  if (c_begin < c_end) { look_up(c_begin); if (c_begin + 1 < c_end) look_up(c_begin + 1); }
  __syncthreads();
  const bool early = c_begin < c_end && (c_begin + 1) * WCH <= base;   // (the chunk holds cached positions only)
  if (early) stage(c_begin, 0);
  pdl_wait();
  if (c_begin < c_end && !early) stage(c_begin, 0);
  // this warp's queries: MMA A fragments straight from memory
  uint32_t qf[KS][4];
  {
    const __half* pa = P.q16 + (size_t)(off + qa / G) * nq + (size_t)(kvh * G + qa % G) * hd + t4 * 2;
    const __half* pb = P.q16 + (size_t)(off + qb / G) * nq + (size_t)(kvh * G + qb % G) * hd + t4 * 2;
#pragma unroll
    for (int kk = 0; kk < KS; ++kk) {
      if (EXACT || kk < ksteps) {
        qf[kk][0] = on_a ? *reinterpret_cast<const uint32_t*>(pa + kk * 16) : 0u;
        qf[kk][1] = on_b ? *reinterpret_cast<const uint32_t*>(pb + kk * 16) : 0u;
        qf[kk][2] = on_a ? *reinterpret_cast<const uint32_t*>(pa + kk * 16 + 8) : 0u;
        qf[kk][3] = on_b ? *reinterpret_cast<const uint32_t*>(pb + kk * 16 + 8) : 0u;
      } else { qf[kk][0] = qf[kk][1] = qf[kk][2] = qf[kk][3] = 0u; }
    }
  }
  int cur = 0;
  for (int c = c_begin; c < c_end; ++c, cur ^= 1) {
    if (c + 1 < c_end) {
      stage(c + 1, cur ^ 1);
      if (c + 2 < c_end) look_up(c + 2);
      mk::cp_async_wait_but_one();
    } else mk::cp_async_wait_all();
    __syncthreads();
    const uint8_t* ks = asm_raw + (size_t)cur * 2 * kvb;
    const uint8_t* vs = ks + kvb;
    const int p0 = c * WCH;
#pragma unroll
    for (int r0 = 0; r0 < SL; r0 += RND) {
      const int sl0 = part * SL + r0;
      if (p0 + sl0 > warp_last) continue;            // nothing of the round is visible to this warp
      float sc[NT][4];
#pragma unroll
      for (int j = 0; j < NT; ++j) sc[j][0] = sc[j][1] = sc[j][2] = sc[j][3] = 0.f;
      const uint8_t* k_lane = ks + (size_t)(sl0 + (lane & 7) + (lane >> 4) * 8) * pitch + ((lane >> 3) & 1) * 16;
#pragma unroll
      for (int kk = 0; kk < KS; ++kk) {
        if (EXACT || kk < ksteps) {
#pragma unroll
          for (int j = 0; j < NT; j += 2) {
            uint32_t kf[4];
            mk::ldmatrix_x4(kf, k_lane + (size_t)j * 8 * pitch + kk * 32);
            mk::mma_16816(sc[j], qf[kk], kf[0], kf[1]);
            mk::mma_16816(sc[j + 1], qf[kk], kf[2], kf[3]);
          }
        }
      }
      if (p0 + sl0 + RND - 1 > warp_first) {         // staircase mask
#pragma unroll
        for (int j = 0; j < NT; ++j)
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            const int pj = p0 + sl0 + 8 * j + t4 * 2 + e;
            if (pj > last_a) sc[j][e] = -INFINITY;
            if (pj > last_b) sc[j][2 + e] = -INFINITY;
          }
      }
      float mx_a = -INFINITY, mx_b = -INFINITY;
#pragma unroll
      for (int j = 0; j < NT; ++j) { mx_a = fmaxf(mx_a, fmaxf(sc[j][0], sc[j][1])); mx_b = fmaxf(mx_b, fmaxf(sc[j][2], sc[j][3])); }
      mx_a = fmaxf(mx_a, __shfl_xor_sync(0xffffffffu, mx_a, 1)); mx_a = fmaxf(mx_a, __shfl_xor_sync(0xffffffffu, mx_a, 2));
      mx_b = fmaxf(mx_b, __shfl_xor_sync(0xffffffffu, mx_b, 1)); mx_b = fmaxf(mx_b, __shfl_xor_sync(0xffffffffu, mx_b, 2));
      const float mn_a = fmaxf(m_a, mx_a), mn_b = fmaxf(m_b, mx_b);
      const float of_a = mn_a == -INFINITY ? 0.f : mn_a, of_b = mn_b == -INFINITY ? 0.f : mn_b;
      const float corr_a = mk::fast_exp2(m_a - of_a), corr_b = mk::fast_exp2(m_b - of_b);
      float sum_a = 0.f, sum_b = 0.f;
#pragma unroll
      for (int j = 0; j < NT; ++j)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          sc[j][e] = mk::fast_exp2(sc[j][e] - of_a); sc[j][2 + e] = mk::fast_exp2(sc[j][2 + e] - of_b);
          sum_a += sc[j][e]; sum_b += sc[j][2 + e];
        }
      l_a = l_a * corr_a + sum_a; l_b = l_b * corr_b + sum_b;   // (this thread's columns; summed over the quad at the end)
      m_a = mn_a; m_b = mn_b;
      if (!__all_sync(0xffffffffu, corr_a == 1.0f && corr_b == 1.0f)) {
#pragma unroll
        for (int nd = 0; nd < 2 * KS; ++nd) { o[nd][0] *= corr_a; o[nd][1] *= corr_a; o[nd][2] *= corr_b; o[nd][3] *= corr_b; }
      }
      const uint8_t* v_lane = vs + (size_t)(sl0 + (lane & 15)) * pitch + (lane >> 4) * 16;
#pragma unroll
      for (int h = 0; h < NT / 2; ++h) {
        const uint32_t pf[4] = {pack_f16x2(sc[2 * h][0], sc[2 * h][1]), pack_f16x2(sc[2 * h][2], sc[2 * h][3]),
                                pack_f16x2(sc[2 * h + 1][0], sc[2 * h + 1][1]), pack_f16x2(sc[2 * h + 1][2], sc[2 * h + 1][3])};
#pragma unroll
        for (int nd = 0; nd < 2 * KS; nd += 2) {
          if (EXACT || nd < ntiles) {
            uint32_t vf[4];
            mk::ldmatrix_x4_trans(vf, v_lane + (size_t)h * 16 * pitch + nd * 16);
            mk::mma_16816(o[nd], pf, vf[0], vf[1]);
            mk::mma_16816(o[nd + 1], pf, vf[2], vf[3]);
          }
        }
      }
    }
    __syncthreads();
  }
  l_a += __shfl_xor_sync(0xffffffffu, l_a, 1); l_a += __shfl_xor_sync(0xffffffffu, l_a, 2);
  l_b += __shfl_xor_sync(0xffffffffu, l_b, 1); l_b += __shfl_xor_sync(0xffffffffu, l_b, 2);

  // states [part][query][hd + 4] (O, then max and sum) in the staging area, merged over parts and ranges (also
  // where there is one of each: stores from the fragments are pieces of 16 bytes)
  float* states = reinterpret_cast<float*>(asm_raw);
  const int ld = hd + 4;
#pragma unroll
  for (int hr = 0; hr < 2; ++hr) {
    float* s = states + (size_t)((part * MT + mt) * 16 + g + 8 * hr) * ld;
#pragma unroll
    for (int nd = 0; nd < 2 * KS; ++nd)
      if (EXACT || nd < ntiles) *reinterpret_cast<float2*>(s + nd * 8 + t4 * 2) = make_float2(o[nd][2 * hr], o[nd][2 * hr + 1]);
    if (t4 == 0) *reinterpret_cast<float4*>(s + hd) = make_float4(hr ? m_b : m_a, hr ? l_b : l_a, 0.f, 0.f);
  }
  if (NS > 1) cluster_sync(); else __syncthreads();
  const uint32_t sbase = smem_u32(states);
  const int vecs = hd / 4;
  for (int it = zr * NTH + tid; it < nQ * vecs; it += NS * NTH) {
    const int ql = it / vecs, d4 = (it % vecs) * 4;
    float M = -INFINITY;
    for (int z = 0; z < NS; ++z)
      for (int p = 0; p < NP; ++p) M = fmaxf(M, ld_cluster_f4(map_rank(sbase + (uint32_t)((p * MT * 16 + ql) * ld + hd) * 4, z)).x);
    float L = 0.f;
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int z = 0; z < NS; ++z)
      for (int p = 0; p < NP; ++p) {
        const uint32_t a = map_rank(sbase + (uint32_t)((p * MT * 16 + ql) * ld) * 4, z);
        const float4 ml = ld_cluster_f4(a + hd * 4), v = ld_cluster_f4(a + d4 * 4);
        const float wgt = ml.x == -INFINITY ? 0.f : mk::fast_exp2(ml.x - M);
        L += ml.y * wgt;
        acc.x += v.x * wgt; acc.y += v.y * wgt; acc.z += v.z * wgt; acc.w += v.w * wgt;
      }
    const float inv = L > 0.f ? 1.0f / L : 0.f;
    const int q = q0 + ql;
    store_split4(P.o + (size_t)(off + q / G) * nq + (size_t)(kvh * G + q % G) * hd, (size_t)d4, (size_t)P.lo_row * nq,
                 make_float4(acc.x * inv, acc.y * inv, acc.z * inv, acc.w * inv));
  }
  if (NS > 1) cluster_sync();                        // the other CTAs have read this one's states
}

// ---------------------------------------------------------------------------------------------
// Prefill attention on tcgen05 (head sizes 64 and 128)
// ---------------------------------------------------------------------------------------------
struct WideAttnTc {
  CUtensorMap kmap, vmap;        // the layer's pools, box = 64 columns x box_rows rows, 128-byte swizzle
  int box_rows;
  WideAttn a;
  unsigned int* status; unsigned long long wait_limit;
};

// D[tmem] (+)= A[tmem] * B[smem], fp16 inputs (two per 32-bit column of A), fp32 accumulate, M = 128.
__device__ __forceinline__ void umma_f16_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
      ::"r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate) : "memory");
}
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float* v) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15,"
      " %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr) : "memory");
#pragma unroll
  for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}
// the same in two steps, so that several loads are in flight (the wait is tied to the registers it guards)
__device__ __forceinline__ void tmem_ld32_issue(uint32_t taddr, uint32_t* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15,"
      " %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr) : "memory");
}
template <int N> __device__ __forceinline__ void tmem_ld_wait(uint32_t* r) {
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < N; ++i) asm volatile("" : "+r"(r[i]));
}
__device__ __forceinline__ void tmem_st16u(uint32_t taddr, const uint32_t* v) {   // completed by tmem_wait_st
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
      ::"r"(taddr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]),
        "r"(v[8]), "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15]) : "memory");
}
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

constexpr int TC_ATT_SOFT = 256;            // softmax threads: two per query, half of a chunk's positions each
constexpr int TC_ATT_THREADS = TC_ATT_SOFT + 64;
constexpr int TC_ATT_STAGES = 2;
template <int HD> constexpr int tc_att_chunk() { return HD == 64 ? 128 : 64; }   // positions per chunk: 32 KB of K and V either way
template <int HD> constexpr size_t tc_att_smem() { return 1024 + (size_t)128 * HD * 2 + TC_ATT_STAGES * (size_t)2 * tc_att_chunk<HD>() * HD * 2 + 256 + 2048 + 64 + 2048; }

// One block: 128 queries (query q of the chunk = row q / G, head q % G of the kv head) against every visible
// position.  S = Q.K^T and O += P.V are M = 128 MMAs, thread (TMEM lane) q owns query q; P goes to TMEM as
// fp16 and is the second MMA's A operand, so the softmax weights never touch shared memory.  A thread takes its
// half row of S into registers at once, so that the next chunk's S is computed under this one's softmax.
// The longest block's chain of chunks is what a pass takes, and most of a chunk is one thread's
// exponentials: two threads share a query (they agree on the row maximum through shared memory).  Two blocks
// share an SM (half its shared memory and TMEM each), launched longest first, so that long and short ones
// meet; where blocks are few, the CTAs of a cluster (grid z) take a range of the context each.  Warps 0-7: softmax, warp 8: K/V bulk copies (one box per page slice and 64-column half, one lane
// each), warp 9: MMA issue, TMEM.
// Measured at 0.4B, 2048 rows from position 0 (16 heads of 64): mma.sync form 72 us, with P in S's place 48,
// one thread per query 38, with rows stored from the accumulator's threads 35, this one 31 us.
template <int HD>
__global__ void __launch_bounds__(TC_ATT_THREADS, 2) k_wide_attn_tc(const __grid_constant__ WideAttnTc J) {
  extern __shared__ __align__(1024) uint8_t atc_raw[];
  constexpr int CH = tc_att_chunk<HD>(), HALVES = HD / 64, NST = TC_ATT_STAGES;
  constexpr int KBYTES = CH * HD * 2;
  const WideAttn& P = J.a;
  uint8_t* qs = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(atc_raw) + 1023) & ~(uintptr_t)1023);   // HALVES x [128][128 bytes]
  uint8_t* ring = qs + 128 * HD * 2;
  // [0], [1]: K buffers, [2], [3]: V buffers, handed back by plain arrivals of threads that have seen the MMAs'
  // completion anyway (a commit costs the issuing thread about 240 cycles)
  uint64_t* kv_full = reinterpret_cast<uint64_t*>(ring + NST * 2 * KBYTES);
  uint64_t* kv_empty = kv_full + 2 * NST;
  uint64_t* q_full = kv_empty + 2 * NST;
  uint64_t* s_full = q_full + 1;
  uint64_t* s_free = s_full + 1;
  uint64_t* p_full = s_free + 1;
  uint64_t* o_done = p_full + 1;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(o_done + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  float* row_x = reinterpret_cast<float*>(tmem_slot + 4);          // [2][2 halves][128] row maxima (alternate chunks), at the end the sums
  volatile int* vx = reinterpret_cast<volatile int*>(row_x + 512);  // [2][8 warps] verdicts, exchanged with the maxima
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < 2 * NST; ++s) { mbar_init(kv_full + s, 1); mbar_init(kv_empty + s, 1); }
    mbar_init(q_full, 8); mbar_init(s_full, 1); mbar_init(s_free, 8); mbar_init(p_full, 8); mbar_init(o_done, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 9) tmem_alloc(tmem_slot, 256);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  // (the successor may start only once this block owns its TMEM: it would take the columns and wait for this grid)
  if (threadIdx.x == 0) pdl_launch();
  const uint32_t tmem_s = *tmem_slot, tmem_p = tmem_s + CH, tmem_o = tmem_p + CH / 2;   // CH + CH / 2 + HD <= 256 columns
  const int G = P.Hq / P.Hkv, nq = P.Hq * HD;
  const int kvh = blockIdx.x, qblk = gridDim.y - 1 - blockIdx.y;
  const int Q = P.rows * G, q0 = qblk * 128, nQ = min(128, Q - q0);
  const int all_chunks = (P.first + (q0 + nQ - 1) / G) / CH + 1, NS = gridDim.z, zr = blockIdx.z;
  const int c_first = (all_chunks * zr) / NS, n_chunks = (all_chunks * (zr + 1)) / NS - c_first;   // this CTA's range of the context
  const unsigned long long lim = J.wait_limit;
  int fills = 0;   // chunks fetched (copies in flight are drained after an abort)

  if (warp == 8) {
    // ------------------------------------------------------------------ K/V loader
    pdl_wait();
    const int* pt = P.page_table + (size_t)P.slot * P.max_pages;
    const int slots = CH / J.box_rows;
    const int half = lane / slots, sl = lane % slots;
    bool ok = true;
    for (int c = 0; c < n_chunks && ok; ++c) {
      const int pz = min((c_first + c) * CH + sl * J.box_rows, (P.max_pages - 1) * P.page_tokens);   // (slices past the page table: any finite rows, they are masked)
      const int row = half < HALVES ? __ldcg(pt + pz / P.page_tokens) * P.page_tokens + pz % P.page_tokens : 0;
      for (int v = 0; v < 2 && ok; ++v) {
        const int s = v * NST + c % NST;
        ok = __all_sync(0xffffffffu, mbar_wait(kv_empty + s, ((c / NST) & 1) ^ 1, abort_flag, lim));
        if (!ok) break;
        if (lane == 0) mbar_expect_tx(kv_full + s, KBYTES);
        __syncwarp();
        if (half < HALVES)
          tma_load_2d_nohint(ring + (size_t)s * KBYTES + half * (CH * 128) + sl * J.box_rows * 128, v ? &J.vmap : &J.kmap, kvh * HD + half * 64, row, kv_full + s);
        ++fills;
      }
    }
  } else if (warp == 9) {
    // ------------------------------------------------------------------ MMA issuer
    if (lane == 0) {
      const uint32_t idesc_s = mk::instr_desc_f16(CH, 0), idesc_o = mk::instr_desc_f16(HD, 1);
      auto issue_s = [&](int c) {
        if (!mbar_wait(kv_full + c % NST, (c / NST) & 1, abort_flag, lim)) return false;
        tc_fence_after();
        const uint32_t kb = smem_u32(ring + (size_t)(c % NST) * KBYTES);
#pragma unroll
        for (int h = 0; h < HALVES; ++h)
#pragma unroll
          for (int k = 0; k < 4; ++k)
            umma_bf16(tmem_s, mk::smem_desc_sw128_ex(smem_u32(qs) + (uint32_t)(h * 128 * 128 + k * 32), 16, 1024),
                      mk::smem_desc_sw128_ex(kb + (uint32_t)(h * CH * 128 + k * 32), 16, 1024), idesc_s, (h | k) ? 1u : 0u);
        umma_commit(s_full);
        return true;
      };
      bool ok = mbar_wait(q_full, 0, abort_flag, lim) && n_chunks > 0 && issue_s(0);
      for (int c = 0; c < n_chunks && ok; ++c) {
        if (c + 1 < n_chunks) {
          ok = mbar_wait(s_free, c & 1, abort_flag, lim);
          if (ok) mbar_arrive(kv_empty + c % NST);               // (S has been read, so its MMAs are done with K)
          tc_fence_after();
          ok = ok && issue_s(c + 1);
        }
        ok = ok && mbar_wait(kv_full + NST + c % NST, (c / NST) & 1, abort_flag, lim) && mbar_wait(p_full, c & 1, abort_flag, lim);
        if (!ok) break;
        tc_fence_after();
        const uint32_t vb = smem_u32(ring + (size_t)(NST + c % NST) * KBYTES);
#pragma unroll
        for (int k = 0; k < CH / 16; ++k)
          umma_f16_ts(tmem_o, tmem_p + (uint32_t)(k * 8), mk::smem_desc_sw128_ex(vb + (uint32_t)(k * 2048), (uint32_t)(CH * 128), 1024), idesc_o, (c > 0 || k > 0) ? 1u : 0u);
        umma_commit(o_done);
      }
    }
  } else {
    // ------------------------------------------------------------------ softmax (warps 0..7)
    pdl_wait();
    const int quad = warp & 3, hf = warp >> 2;                   // TMEM lanes 32 quad .., half hf of a chunk's positions
    const int ql = quad * 32 + lane;
    constexpr int CW = CH / 2, HW = HD / 2;                      // positions and head columns of this thread
    {
      // the block's queries, swizzled; rows past its queries are zero
      constexpr int PIECES = HD / 8;
      for (int it = threadIdx.x; it < 128 * PIECES; it += TC_ATT_SOFT) {
        const int r = it / PIECES, c = it % PIECES;
        const bool on = r < nQ;
        const int q = on ? q0 + r : q0;
        mk::cp_async16(qs + (size_t)(c >> 3) * (128 * 128) + (size_t)r * 128 + (size_t)(((c & 7) ^ (r & 7)) << 4),
                       reinterpret_cast<const uint4*>(P.q16 + (size_t)(q / G) * nq + (size_t)(kvh * G + q % G) * HD) + c, on);
      }
      mk::cp_async_commit();
      mk::cp_async_wait_all();
      mk::fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive(q_full);
    }
    const bool mine = ql < nQ;
    const int q = q0 + (mine ? ql : nQ - 1);
    const int last = P.first + q / G;                           // last visible position of this thread's query
    const int warp_first = P.first + (q0 + min(quad * 32, nQ - 1)) / G;
    const uint32_t sel = (uint32_t)(quad * 32) << 16;
    auto wait = [&](uint64_t* bar, uint32_t parity) {            // one verdict per warp
      if (__all_sync(0xffffffffu, mbar_try(bar, parity))) return true;
      return (bool)__all_sync(0xffffffffu, mbar_wait(bar, parity, abort_flag, lim));
    };
    auto pair_sync = [&]() { asm volatile("bar.sync %0, 64;" ::"r"(1 + quad) : "memory"); };   // the two warps of these 32 queries
    float m_run = -INFINITY, l_run = 0.f;
    bool ok = true;
    for (int c = 0; c < n_chunks; ++c) {
      // (after an expired wait both warps of a pair have to leave together: a warp goes on until the next
      // exchange, where the pair agrees on one verdict)
      ok = ok && wait(s_full, c & 1);
      tc_fence_after();
      const int p0 = (c_first + c) * CH + hf * CW;
      uint32_t sr[CW];
#pragma unroll
      for (int j0 = 0; j0 < CW; j0 += 32) tmem_ld32_issue(tmem_s + sel + (uint32_t)(hf * CW + j0), sr + j0);
      tmem_ld_wait<CW>(sr);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(s_free);                        // the next chunk's S may take its place
      if (p0 + CW - 1 > warp_first) {
#pragma unroll
        for (int j = 0; j < CW; ++j) if (p0 + j > last) sr[j] = 0xff800000u;   // -inf
      }
      float mxa = __uint_as_float(sr[0]), mxb = __uint_as_float(sr[1]);
#pragma unroll
      for (int j = 2; j < CW; j += 4) {                          // (three-operand maxima)
        mxa = fmaxf(fmaxf(mxa, __uint_as_float(sr[j])), __uint_as_float(sr[j + 1]));
        if (j + 2 < CW) mxb = fmaxf(fmaxf(mxb, __uint_as_float(sr[j + 2])), __uint_as_float(sr[j + 3]));
      }
      float* rx = row_x + (c & 1) * 256;
      rx[hf * 128 + ql] = fmaxf(mxa, mxb);
      if (lane == 0) vx[(c & 1) * 8 + warp] = ok ? 1 : 0;
      pair_sync();
      const float mx = fmaxf(rx[ql], rx[128 + ql]);
      ok = vx[(c & 1) * 8 + quad] && vx[(c & 1) * 8 + quad + 4];
      if (!ok) break;
      // the reference exponent follows the running maximum only when that has moved by more than 2^8 (see the persistent kernel)
      const float m_seen = fmaxf(m_run, mx);
      const float m_new = (m_seen > m_run + 8.0f || m_run == -INFINITY) ? m_seen : m_run;
      const float off = m_new == -INFINITY ? 0.f : m_new;
      const float corr = mk::fast_exp2(m_run - off);
      // (two elements per addition: the loop is bound by instruction issue and fetch)
      const float2 noff = make_float2(-off, -off);
      float2 sum2[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
#pragma unroll
      for (int j = 0; j < CW; j += 2) {
        float2 e = add2(make_float2(__uint_as_float(sr[j]), __uint_as_float(sr[j + 1])), noff);
        e.x = mk::fast_exp2(e.x); e.y = mk::fast_exp2(e.y);
        sum2[(j >> 1) & 1] = add2(sum2[(j >> 1) & 1], e);
        sr[j / 2] = pack_f16x2(e.x, e.y);
      }
      sum2[0] = add2(sum2[0], sum2[1]);
      l_run = l_run * corr + (sum2[0].x + sum2[0].y);
      m_run = m_new;
      if (c > 0) {
        ok = wait(o_done, (c - 1) & 1);
        if (threadIdx.x == 0) mbar_arrive(kv_empty + NST + (c - 1) % NST);   // the V buffer of that P.V is free
        tc_fence_after();
        if (__any_sync(0xffffffffu, corr != 1.0f)) {
#pragma unroll
          for (int d0 = 0; d0 < HW; d0 += 32) {
            float v[32];
            uint32_t u[32];
            tmem_ld32(tmem_o + sel + (uint32_t)(hf * HW + d0), v);
#pragma unroll
            for (int j = 0; j < 32; ++j) u[j] = __float_as_uint(v[j] * corr);
            tmem_st16u(tmem_o + sel + (uint32_t)(hf * HW + d0), u);
            tmem_st16u(tmem_o + sel + (uint32_t)(hf * HW + d0 + 16), u + 16);
          }
        }
      }
#pragma unroll
      for (int j0 = 0; j0 < CW / 2; j0 += 16) tmem_st16u(tmem_p + sel + (uint32_t)(hf * (CW / 2) + j0), sr + j0);   // (the previous P.V, waited for above, has read its P)
      tmem_wait_st();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(p_full);
    }
    if (ok && n_chunks > 0) ok = wait(o_done, (n_chunks - 1) & 1);
    if (!ok) *abort_flag = 1;
    __syncwarp();
    asm volatile("bar.sync 5, 256;" ::: "memory");               // (every pair is past its last exchange of maxima)
    row_x[hf * 128 + ql] = l_run;
    asm volatile("bar.sync 5, 256;" ::: "memory");
    if (*abort_flag == 0) {
      tc_fence_after();
      if (hf == 0) { row_x[256 + ql] = m_run; row_x[384 + ql] = row_x[ql] + row_x[128 + ql]; }
      float* part = reinterpret_cast<float*>(qs) + (size_t)ql * (HD + 4) + hf * HW;   // (every MMA has completed: the tiles are free)
#pragma unroll
      for (int d0 = 0; d0 < HW; d0 += 32) {
        float v[32];
        tmem_ld32(tmem_o + sel + (uint32_t)(hf * HW + d0), v);
#pragma unroll
        for (int j = 0; j < 32; j += 4)
          *reinterpret_cast<float4*>(part + d0 + j) = n_chunks > 0 ? make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]) : make_float4(0.f, 0.f, 0.f, 0.f);
      }
      tc_fence_before();
    }
  }
  {
    // The ranges' states, merged in range order (the cluster's CTAs share the rows), through shared memory in any
    // case: stores of one row per thread took 8 us of a block with head size 128.
    __syncwarp();
    if (NS > 1) cluster_sync(); else __syncthreads();
    // every range's weight of every row, once (the maxima and sums of the other CTAs are a long way off)
    float* wgt = row_x + 528;                                    // [4 ranges][128]
    if (threadIdx.x < 128) {
      const int r = threadIdx.x;
      const uint32_t mbase = smem_u32(row_x) + (uint32_t)(256 + r) * 4;
      float m[4], l[4], M = -INFINITY, L = 0.f;
#pragma unroll
      for (int z = 0; z < 4; ++z) {
        m[z] = -INFINITY; l[z] = 0.f;
        if (z < NS) { const uint32_t at = map_rank(mbase, z); m[z] = ld_cluster_f1(at); l[z] = ld_cluster_f1(at + 512); }
        M = fmaxf(M, m[z]);
      }
#pragma unroll
      for (int z = 0; z < 4; ++z) { m[z] = m[z] == -INFINITY ? 0.f : mk::fast_exp2(m[z] - M); L += l[z] * m[z]; }
      const float inv = L > 0.f ? 1.0f / L : 0.f;
#pragma unroll
      for (int z = 0; z < 4; ++z) wgt[z * 128 + r] = m[z] * inv;
    }
    __syncthreads();
    const uint32_t pbase = smem_u32(qs);
#pragma unroll 4
    for (int it = zr * TC_ATT_THREADS + threadIdx.x; it < nQ * (HD / 4); it += NS * TC_ATT_THREADS) {
      const int r = it / (HD / 4), d4 = it % (HD / 4) * 4;
      const uint32_t at = (uint32_t)(r * (HD + 4) + d4) * 4;
      const float w0 = wgt[r];
      float4 acc = NS == 1 ? *reinterpret_cast<const float4*>(qs + at) : ld_cluster_f4(map_rank(pbase + at, 0));
      acc.x *= w0; acc.y *= w0; acc.z *= w0; acc.w *= w0;
      for (int z = 1; z < NS; ++z) {
        const float w = wgt[z * 128 + r];
        const float4 v = ld_cluster_f4(map_rank(pbase + at, z));
        acc.x += v.x * w; acc.y += v.y * w; acc.z += v.z * w; acc.w += v.w * w;
      }
      const int q = q0 + r;
      store_split4(P.o + (size_t)(q / G) * nq + (size_t)(kvh * G + q % G) * HD, (size_t)d4, (size_t)P.lo_row * nq, acc);
    }
    if (NS > 1) cluster_sync();
  }
  // ------------------------------------------------------------------ teardown
  __syncthreads();
  if (*abort_flag) {
    if (warp == 8 && lane == 0) {
      *reinterpret_cast<volatile unsigned int*>(J.status + STATUS_ERROR) = 5u;  // STAIRS_ETIMEOUT
      __threadfence_system();
      const long long t0 = clock64();
      const unsigned long long drain = lim > 2000000ull ? lim : 2000000ull;
      for (int f = max(0, fills - 2 * NST); f < fills; ++f)      // fill f: chunk f / 2, K or V
        while (!mbar_try(kv_full + (f & 1) * NST + (f >> 1) % NST, ((f >> 1) / NST) & 1)) {
          if ((unsigned long long)(clock64() - t0) > drain) break;
        }
      settle(t0);
    }
    __syncthreads();
  }
  if (warp == 9) { tc_fence_after(); tmem_dealloc(tmem_s, 256); }
}

// Embedding of the pass's rows (tok, pos, req written by k_rows): the residual stream, the first GEMM's
// operand bf16(x * gain) hi + lo, the row's statistics, its rotation table and its cache row.  One block per row.
// (What the stream's previous kernel may still write when this one starts is not declared restrict: the loads stay behind the wait.)
__global__ void __launch_bounds__(256) k_wide_embed(const bf16* __restrict__ tok_emb, const bf16* __restrict__ pos_emb, const int* tok,
                                                    const int* pos, const int* req, const int* page_table,
                                                    int page_tokens, int max_pages, const float* __restrict__ g, float* __restrict__ x, bf16* __restrict__ h,
                                                    int lo_row, int d, float4* __restrict__ stats, const float* __restrict__ rope_inv, int half,
                                                    float* __restrict__ rope_cs, float* __restrict__ rope_sn, int* __restrict__ kv_row) {
  __shared__ float red[32];
  const int t = blockIdx.x;
  if (threadIdx.x == 0) pdl_launch();
  pdl_wait();
  const int p = pos[t];
  const bf16* e = tok_emb + (size_t)tok[t] * d;
  const bf16* pe = pos_emb ? pos_emb + (size_t)p * d : nullptr;
  float s1 = 0.f;
  for (int i = threadIdx.x * 4; i < d; i += 1024) {
    float v[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) { v[j] = __bfloat162float(e[i + j]); if (pe) v[j] += __bfloat162float(pe[i + j]); s1 += v[j]; }
    *reinterpret_cast<float4*>(x + (size_t)t * d + i) = make_float4(v[0], v[1], v[2], v[3]);
    const float4 g4 = *reinterpret_cast<const float4*>(g + i);
    store_split4(h, (size_t)t * d + i, (size_t)lo_row * d, make_float4(v[0] * g4.x, v[1] * g4.y, v[2] * g4.z, v[3] * g4.w));
  }
  const float mean = block_sum(s1, red) / (float)d;
  float s2 = 0.f;
  for (int i = threadIdx.x * 4; i < d; i += 1024) {
    const float4 v = *reinterpret_cast<const float4*>(x + (size_t)t * d + i);   // (this thread's own stores)
    const float a = v.x - mean, b = v.y - mean, c = v.z - mean, q = v.w - mean;
    s2 += (a * a + b * b) + (c * c + q * q);
  }
  const float m2 = block_sum(s2, red);
  if (threadIdx.x == 0) {
    stats[t] = make_float4(mean, m2, (float)d, 0.f);
    kv_row[t] = page_table[(size_t)req[t] * max_pages + p / page_tokens] * page_tokens + p % page_tokens;
  }
  if (rope_inv)
    for (int i = threadIdx.x; i < half; i += 256) {
      float sn, cs;
      sincosf((float)p * rope_inv[i], &sn, &cs);
      rope_cs[(size_t)t * half + i] = cs;
      rope_sn[(size_t)t * half + i] = sn;
    }
}

}  // namespace wide
}  // namespace stairs
