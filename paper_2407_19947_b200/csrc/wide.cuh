// Passes over many rows (prefill chunks, serving batches of more than 64 stair rows): one launch per
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
// Warp roles (192 threads): warp 0 TMA producer, warp 1 MMA issuer and TMEM owner, warps 2-5 epilogue
// (one TMEM lane quadrant each).  Two accumulators in TMEM let a tile's epilogue run under the next
// tile's MMAs.  Launches are chained with programmatic dependent launch: a kernel sets itself up and
// fetches its first weight tiles while its predecessor finishes, and touches what the predecessor wrote
// only after griddepcontrol.wait.  All waits are bounded like everywhere in this library.
#pragma once
#include "megakernel.cuh"

namespace stairs {
namespace wide {

using namespace tc;
using mk::store_split4;
using mk::pack_f16x2;
using mk::tma_load_2d_nohint;

constexpr int WM = 128;                    // rows per CTA
constexpr int WTHREADS = 192;
constexpr int W_MAX_STAGES = 8;
constexpr int A_BYTES = WM * BK * 2;       // one part (hi or lo) of the activation tile
constexpr int ST_LD = 36;                  // row pitch (floats) of a warp's 32 x 32 exchange tile
constexpr int ST_BYTES = 4 * 32 * ST_LD * 4;

enum WEpi { W_ADD = 0, W_GELU = 1, W_SWIGLU = 2, W_QKV = 3, W_LMHEAD = 4 };

struct WideJob {
  CUtensorMap x_map;        // [2 * lo_row rows][K]; box 64 x x_box
  CUtensorMap w_map[3];     // box 64 x b_box rows
  int n_src, src_tiles[3], src_rows[3];
  int src0;                 // W_QKV: first source present (0: q, k, v; 1: k and v only)
  int x_box, b_box, b_boxes;   // b_boxes: weight boxes per CTA and k-block (2: a 32-row gate box and its up box)
  int T, TN, n_tiles, m_tiles, kblocks, splits, stages;
  int lo_row;               // rows between the hi and the lo part of every bf16 operand
  int epi;
  int N, ldo;               // output features (SwiGLU: of one matrix), leading dimension of the output
  int gsz;                  // SwiGLU: width of a gate block (its up block follows)
  float* out_f32;           // W_ADD: the residual stream; W_LMHEAD: logits (may be null)
  bf16* out_act;            // W_GELU / W_SWIGLU: ff; W_ADD with next_g: the next operand
  const float* next_g;
  // folded normalisation of the operand (see the persistent kernel)
  int norm_in, norm_kind, d; float eps;
  const float4* stats_in; int stat_tiles_in;    // (mean, M2, count) per row and column tile of x
  float4* stats_out;                            // W_ADD with next_g: [row][n_tiles]
  const float* u; const float* c; int u_off[3];   // (u_off: first entry of each source)
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
      : "r"(taddr));
#pragma unroll
  for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

// ---------------------------------------------------------------------------------------------
// The GEMM
// ---------------------------------------------------------------------------------------------
template <int CG>
__global__ void __launch_bounds__(WTHREADS, 1) k_wide_gemm(const __grid_constant__ WideJob job) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  const int TN = job.TN, TNc = TN / CG, stages = job.stages, S = job.splits;
  const int stage_bytes = 2 * A_BYTES + TNc * BK * 2;
  uint8_t* tail = smem + (size_t)stages * stage_bytes;
  float* stile = reinterpret_cast<float*>(tail);                     // [4 warps][32][ST_LD]
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
  uint32_t tmem_cols = 32;
  while ((int)tmem_cols < 2 * TN) tmem_cols <<= 1;

  if (threadIdx.x == 0) {
    for (int s = 0; s < stages; ++s) { mbar_init(full + s, 1); mbar_init(empty + s, 1); }
    mbar_init(acc_full + 0, 1); mbar_init(acc_full + 1, 1);
    mbar_init(acc_empty + 0, 4 * CG); mbar_init(acc_empty + 1, 4 * CG);
    *abort_flag = 0; *verdict = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) w_alloc<CG>(tmem_slot, tmem_cols);
  tc_fence_before();
  if (CG == 2) cluster_sync(); else __syncthreads();
  tc_fence_after();
  if (CG == 2) __syncthreads();
  const uint32_t tmem_base = *tmem_slot;
  if (threadIdx.x == 0) pdl_launch();
  int issued = 0, p_stage = 0;
  uint32_t p_phase = 0;
  auto k_begin = [&](int s) { return (job.kblocks * s) / S; };

  if (warp == 0) {
    // ------------------------------------------------------------------ TMA producer
    if (lane == 0) {
      const uint64_t pol_w = policy_evict_first(), pol_x = policy_evict_last();
      const uint32_t tx = (uint32_t)(CG * (2 * job.x_box * BK * 2 + TNc * BK * 2));   // both CTAs' bytes
      auto load_w = [&](int tile, int kb, int stage) {
        uint8_t* dst = smem + (size_t)stage * stage_bytes + 2 * A_BYTES;
        int s = 0, local = tile;
        while (s + 1 < job.n_src && local >= job.src_tiles[s]) { local -= job.src_tiles[s]; ++s; }
        if (job.b_boxes == 2) {   // 32 gate rows and their 32 up rows, half a packed 64 + 64 tile
          const int row = (local >> 1) * 128 + (local & 1) * 32;
          w_tma<CG>(dst, &job.w_map[0], kb * BK, row, full + stage, pol_w);
          w_tma<CG>(dst + 32 * BK * 2, &job.w_map[0], kb * BK, row + 64, full + stage, pol_w);
        } else {
          w_tma<CG>(dst, &job.w_map[s], kb * BK, local * TN + rank * TNc, full + stage, pol_w);
        }
      };
      int stage = 0; uint32_t phase = 0;
      // the first weight tiles depend on nothing: fetched before the predecessor's results are waited for
      int ahead = 0;
      if (cid < units) {
        const int s0 = cid % S, nt0 = (cid / S) / job.m_tiles;
        const int kb0 = k_begin(s0), kb1 = k_begin(s0 + 1);
        for (; ahead < stages && ahead < kb1 - kb0; ++ahead) {
          if (rank == 0) mbar_expect_tx(full + ahead, tx);
          load_w(nt0, kb0 + ahead, ahead);
        }
      }
      pdl_wait();
      bool ok = true;
      for (int u = cid; u < units && ok; u += G) {
        const int s = u % S, tile = u / S, nt = tile / job.m_tiles, mt = tile % job.m_tiles;
        const int x_row = (mt * CG + rank) * WM;
        const int kb1 = k_begin(s + 1);
        for (int kb = k_begin(s); kb < kb1; ++kb) {
          if (issued >= ahead) {
            if (!mbar_wait(empty + stage, phase ^ 1, abort_flag, job.wait_limit)) { ok = false; break; }
            if (rank == 0) mbar_expect_tx(full + stage, tx);
            load_w(nt, kb, stage);
          }
          uint8_t* dst = smem + (size_t)stage * stage_bytes;
          w_tma<CG>(dst, &job.x_map, kb * BK, x_row, full + stage, pol_x);
          w_tma<CG>(dst + A_BYTES, &job.x_map, kb * BK, job.lo_row + x_row, full + stage, pol_x);
          ++issued;
          if (++stage == stages) { stage = 0; phase ^= 1; }
          p_stage = stage; p_phase = phase;
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
          const uint64_t hi = smem_desc_sw128(a), lo = smem_desc_sw128(a + A_BYTES), w = smem_desc_sw128(a + 2 * A_BYTES);
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
    // ------------------------------------------------------------------ epilogue (warps 2..5)
    const int quad = warp & 3, et = threadIdx.x - 64;
    float* st = stile + (size_t)quad * 32 * ST_LD;
    const int tr = lane >> 3, tc4 = (lane & 7) * 4;    // exchange-tile mapping: row 4 i + tr, four columns from tc4
    int buf = 0; uint32_t acc_bits = 0;
    pdl_wait();
    for (int u = cid; u < units; u += G) {
      const int sp = u % S, tile = u / S, nt = tile / job.m_tiles, mt = tile % job.m_tiles;
      const int row0 = (mt * CG + rank) * WM + quad * 32, row = row0 + lane;
      const bool row_on = row < job.T;
      int src = 0, local = nt;
      while (src + 1 < job.n_src && local >= job.src_tiles[src]) { local -= job.src_tiles[src]; ++src; }
      const int col0 = local * TN;                      // first weight row of the tile in its source
      // what the epilogue reads from memory is requested before the accumulator is waited for
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
      float4 xq[8];
      auto load_x = [&](int c0) {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const int r = row0 + 4 * i + tr;
          xq[i] = (r < job.T && col0 + c0 < job.N) ? __ldcg(reinterpret_cast<const float4*>(job.out_f32 + (size_t)r * job.ldo + col0 + c0 + tc4))
                                                    : make_float4(0.f, 0.f, 0.f, 0.f);
        }
      };
      if (job.epi == W_ADD && S == 1) load_x(0);
      bool ok = mbar_wait(acc_full + buf, (acc_bits >> buf) & 1u, abort_flag, job.wait_limit);
      ok = __all_sync(0xffffffffu, ok);
      if (S > 1) {   // the split tiles' barriers below want one verdict for the whole group
        if (!ok) *abort_flag = 1;
        epi_bar_sync();
        if (et == 0) *verdict = *abort_flag ? 0 : 1;
        epi_bar_sync();
        ok = *verdict != 0;
      }
      if (!ok) break;
      acc_bits ^= 1u << buf;
      tc_fence_after();
      const uint32_t taddr = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)buf * (tmem_cols / 2);
      bool finish = true;
      const float* parts = nullptr;
      const size_t part_stride = (size_t)TN * WM;
      if (S > 1) {
        // a K range of the tile: park it ([4 columns][row] vectors), the last arriver adds the ranges in K order
        float* base = job.partial + (size_t)tile * S * part_stride;
        parts = base;
        float* mine = base + (size_t)sp * part_stride + (size_t)(quad * 32 + lane) * 4;
        for (int c0 = 0; c0 < TN; c0 += 8) {
          float v[8];
          tmem_ld8(taddr + (uint32_t)c0, v);
          if (row_on) {
            *reinterpret_cast<float4*>(mine + (size_t)c0 * WM) = make_float4(v[0], v[1], v[2], v[3]);
            *reinterpret_cast<float4*>(mine + (size_t)(c0 + 4) * WM) = make_float4(v[4], v[5], v[6], v[7]);
          }
        }
        __threadfence();
        epi_bar_sync();
        if (et == 0) {
          const int old = atomicAdd(job.counters + tile, 1);
          if (old == S - 1) job.counters[tile] = 0;
          *verdict = old == S - 1 ? 2 : 1;
        }
        epi_bar_sync();
        finish = *verdict == 2;
        if (finish) { __threadfence(); if (job.epi == W_ADD) load_x(0); }
      }
      // n consecutive accumulator columns of this thread's row
      auto acc8 = [&](int c0, float* v) {
        if (S == 1) { tmem_ld8(taddr + (uint32_t)c0, v); return; }
        const float* p0 = parts + (size_t)(quad * 32 + lane) * 4 + (size_t)c0 * WM;
#pragma unroll
        for (int j = 0; j < 8; ++j) v[j] = 0.f;
        if (row_on)
          for (int s2 = 0; s2 < S; ++s2) {
            const float4 a = __ldcg(reinterpret_cast<const float4*>(p0 + s2 * part_stride)), b = __ldcg(reinterpret_cast<const float4*>(p0 + s2 * part_stride + 4 * WM));
            v[0] += a.x; v[1] += a.y; v[2] += a.z; v[3] += a.w; v[4] += b.x; v[5] += b.y; v[6] += b.z; v[7] += b.w;
          }
      };
      auto acc32 = [&](int c0, float* v) {
        if (S == 1) { tmem_ld32(taddr + (uint32_t)c0, v); return; }
        const float* p0 = parts + (size_t)(quad * 32 + lane) * 4 + (size_t)c0 * WM;
#pragma unroll
        for (int j = 0; j < 32; ++j) v[j] = 0.f;
        if (row_on)
          for (int s2 = 0; s2 < S; ++s2) {
            float4 a[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) a[j] = __ldcg(reinterpret_cast<const float4*>(p0 + s2 * part_stride + (size_t)(4 * j) * WM));
#pragma unroll
            for (int j = 0; j < 8; ++j) { v[4 * j] += a[j].x; v[4 * j + 1] += a[j].y; v[4 * j + 2] += a[j].z; v[4 * j + 3] += a[j].w; }
          }
      };
      // folded normalisation of a column of weight row n (u and c are the same for all lanes)
      auto normed = [&](float v, int n) { return job.u ? rs * (v - mu * __ldg(job.u + n)) + __ldg(job.c + n) : rs * v; };
      auto to_tile = [&](const float* v) {
        __syncwarp();
#pragma unroll
        for (int j = 0; j < 8; ++j) *reinterpret_cast<float4*>(st + lane * ST_LD + 4 * j) = make_float4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
        __syncwarp();
      };
      auto store_act = [&](int out_col) {   // the exchange tile as bf16 hi + lo, 64 contiguous bytes per row and part
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const int r = row0 + 4 * i + tr;
          if (r < job.T && out_col + tc4 < job.N)
            store_split4(job.out_act, (size_t)r * job.ldo + out_col + tc4, (size_t)job.lo_row * job.ldo, *reinterpret_cast<const float4*>(st + (4 * i + tr) * ST_LD + tc4));
        }
      };
      if (finish) {
        if (job.epi == W_ADD) {
          // residual update, the next GEMM's operand bf16(x * gain), and this tile's row statistics (shifted
          // sums: the shift is the row's first value of the tile)
          float s1[8], s2[8], sh[8];
#pragma unroll
          for (int i = 0; i < 8; ++i) { s1[i] = s2[i] = sh[i] = 0.f; }
          for (int c0 = 0; c0 < TN && col0 + c0 < job.N; c0 += 32) {
            float v[32];
            acc32(c0, v);
            to_tile(v);
            const int col = col0 + c0 + tc4;
            const float4 g4 = job.next_g ? __ldg(reinterpret_cast<const float4*>(job.next_g + col)) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
            for (int i = 0; i < 8; ++i) {
              const int r = row0 + 4 * i + tr;
              const float4 a = *reinterpret_cast<const float4*>(st + (4 * i + tr) * ST_LD + tc4);
              const float4 x4 = make_float4(xq[i].x + a.x, xq[i].y + a.y, xq[i].z + a.z, xq[i].w + a.w);
              if (r < job.T) {
                *reinterpret_cast<float4*>(job.out_f32 + (size_t)r * job.ldo + col) = x4;
                if (job.next_g)
                  store_split4(job.out_act, (size_t)r * job.ldo + col, (size_t)job.lo_row * job.ldo, make_float4(x4.x * g4.x, x4.y * g4.y, x4.z * g4.z, x4.w * g4.w));
              }
              if (c0 == 0) sh[i] = __shfl_sync(0xffffffffu, x4.x, lane & 24);
              const float d0 = x4.x - sh[i], d1 = x4.y - sh[i], d2 = x4.z - sh[i], d3 = x4.w - sh[i];
              s1[i] += (d0 + d1) + (d2 + d3);
              s2[i] += (d0 * d0 + d1 * d1) + (d2 * d2 + d3 * d3);
            }
            if (c0 + 32 < TN) load_x(c0 + 32);
          }
          if (job.next_g) {
            const float cnt = (float)min(TN, job.N - col0);
#pragma unroll
            for (int i = 0; i < 8; ++i) {
#pragma unroll
              for (int o = 1; o < 8; o <<= 1) { s1[i] += __shfl_xor_sync(0xffffffffu, s1[i], o); s2[i] += __shfl_xor_sync(0xffffffffu, s2[i], o); }
              const int r = row0 + 4 * i + tr;
              const float m = s1[i] / cnt;
              if ((lane & 7) == 0 && r < job.T) job.stats_out[(size_t)r * job.n_tiles + nt] = make_float4(sh[i] + m, fmaxf(s2[i] - s1[i] * m, 0.f), cnt, 0.f);
            }
          }
        } else if (job.epi == W_GELU) {
          for (int c0 = 0; c0 < TN && col0 + c0 < job.N; c0 += 32) {
            float v[32];
            acc32(c0, v);
#pragma unroll
            for (int j = 0; j < 32; ++j) v[j] = gelu_erf(normed(v[j], col0 + c0 + j));
            to_tile(v);
            store_act(col0 + c0);
          }
        } else if (job.epi == W_SWIGLU) {
          const int gsz = job.gsz, out0 = local * (TN / 2);
          for (int b = 0; b < TN; b += 2 * gsz)
            for (int c0 = 0; c0 < gsz; c0 += 32) {
              const int oc = out0 + b / 2 + c0;
              if (oc >= job.N) break;
              float v[32], w[32];
              acc32(b + c0, v);
              acc32(b + gsz + c0, w);
#pragma unroll
              for (int j = 0; j < 32; ++j) v[j] = silu_f(normed(v[j], oc + j)) * normed(w[j], job.N + oc + j);
              to_tile(v);
              store_act(oc);
            }
        } else if (job.epi == W_LMHEAD) {
          unsigned long long key = 0ull;
          for (int c0 = 0; c0 < TN && col0 + c0 < job.N; c0 += 32) {
            float v[32];
            acc32(c0, v);
#pragma unroll
            for (int j = 0; j < 32; ++j) {
              const int n = col0 + c0 + j;
              v[j] = normed(v[j], min(n, job.N - 1));
              const unsigned long long k2 = argmax_key(v[j], (uint32_t)n);
              if (n < job.N && k2 > key) key = k2;
            }
            if (job.out_f32) {
              to_tile(v);
              const int n = col0 + c0 + lane;
              for (int r = 0; r < 32 && row0 + r < job.T; ++r)
                if (n < job.N) job.out_f32[(size_t)(row0 + r) * job.ldo + n] = st[r * ST_LD + lane];
            }
          }
          if (row_on && key) atomicMax(job.keys + row, key);
        } else {   // W_QKV: rotate and scale q, rotate k; fp16 to the query buffer and the cache
          const int hd = job.hd, half = hd / 2, width = job.src_rows[src], part = src + job.src0;   // part 0: q, 1: k, 2: v
          const int u0 = job.u_off[src];
          const int rr = row_on ? row : 0;
          __half* dst = (part == 0 ? job.q16 + (size_t)rr * width : (part == 1 ? job.kc : job.vc) + (size_t)__ldcg(job.kv_row + rr) * width) + col0;
          const float qs = part == 0 ? job.qscale : 1.0f;
          const bool rot = job.rope && part < 2;
          for (int h0 = 0; h0 < TN && col0 + h0 < width; h0 += hd)
            for (int i0 = 0; i0 < half; i0 += 8) {
              float lo[8], hi[8];
              acc8(h0 + i0, lo);
              acc8(h0 + half + i0, hi);
#pragma unroll
              for (int j = 0; j < 8; ++j) {
                lo[j] = normed(lo[j], u0 + col0 + h0 + i0 + j);
                hi[j] = normed(hi[j], u0 + col0 + h0 + half + i0 + j);
              }
              if (rot) {
                const float4* cp = reinterpret_cast<const float4*>(job.rope_cs + (size_t)rr * half + i0);
                const float4* sp4 = reinterpret_cast<const float4*>(job.rope_sn + (size_t)rr * half + i0);
                const float4 ca = __ldcg(cp), cb = __ldcg(cp + 1), sa = __ldcg(sp4), sb = __ldcg(sp4 + 1);
                const float cs[8] = {ca.x, ca.y, ca.z, ca.w, cb.x, cb.y, cb.z, cb.w}, sn[8] = {sa.x, sa.y, sa.z, sa.w, sb.x, sb.y, sb.z, sb.w};
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                  const float l = lo[j], h = hi[j];
                  lo[j] = l * cs[j] - h * sn[j]; hi[j] = h * cs[j] + l * sn[j];
                }
              }
              if (row_on) {
                *reinterpret_cast<uint4*>(dst + h0 + i0) = make_uint4(pack_f16x2(lo[0] * qs, lo[1] * qs), pack_f16x2(lo[2] * qs, lo[3] * qs),
                                                                      pack_f16x2(lo[4] * qs, lo[5] * qs), pack_f16x2(lo[6] * qs, lo[7] * qs));
                *reinterpret_cast<uint4*>(dst + h0 + half + i0) = make_uint4(pack_f16x2(hi[0] * qs, hi[1] * qs), pack_f16x2(hi[2] * qs, hi[3] * qs),
                                                                             pack_f16x2(hi[4] * qs, hi[5] * qs), pack_f16x2(hi[6] * qs, hi[7] * qs));
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
    }
    __syncthreads();
  }
  if (CG == 2) cluster_sync();   // neither CTA leaves while the other may still use its shared memory or barriers
  if (warp == 1) { tc_fence_after(); w_dealloc<CG>(tmem_base, tmem_cols); }
}

inline size_t gemm_smem(int TN, int CG, int stages) {
  return 1024 + (size_t)stages * (2 * A_BYTES + (size_t)(TN / CG) * BK * 2) + ST_BYTES + (2 * W_MAX_STAGES + 4) * 8 + 64;
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
// <4, 1..4> requests with few query rows, whose warps split the positions instead.  Long contexts of few
// blocks are cut over a cluster of up to 8 CTAs (grid z); slices and ranges are merged at the end through
// (distributed) shared memory in a fixed order.  Chunks are staged by 16-byte asynchronous copies, the
// next one under the current one's MMAs.
// EXACT: hd == 16 * KS (loops without guards).
template <int KS, bool EXACT, int NW, int MT>
__global__ void __launch_bounds__(NW * 32, (KS <= 5 && NW == 8) ? 2 : 1) k_wide_attn(const __grid_constant__ WideAttn P) {
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
  pdl_wait();
  int slot, base, R, off;
  const int i_req = blockIdx.x / P.n_qblk, kvh = blockIdx.y;
  int qblk = blockIdx.x % P.n_qblk;
  if (P.val_req) {
    slot = P.val_req[i_req]; R = P.val_k[i_req] + 1; off = P.val_off[i_req]; base = P.n_seq[slot] - 1;
  } else { slot = P.slot; R = P.rows; off = 0; base = P.first; qblk = P.n_qblk - 1 - qblk; }   // (the longest blocks first)
  const int Q = R * G, q0 = qblk * MT * 16;
  if (q0 >= Q) return;                              // (uniform over the cluster)
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

  // this warp's queries: MMA A fragments straight from memory
  const int ql_a = mt * 16 + g, ql_b = ql_a + 8;
  const bool on_a = ql_a < nQ, on_b = ql_b < nQ;
  const int qa = q0 + (on_a ? ql_a : 0), qb = q0 + (on_b ? ql_b : 0);
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
  const int last_a = on_a ? base + qa / G : -1, last_b = on_b ? base + qb / G : -1;
  const int warp_first = base + (q0 + mt * 16) / G;                                       // first query's last visible position
  const int warp_last = mt * 16 < nQ ? base + (q0 + min(mt * 16 + 15, nQ - 1)) / G : -1;  // (-1: no queries)
  float m_a = -INFINITY, m_b = -INFINITY, l_a = 0.f, l_b = 0.f;
  float o[2 * KS][4];
#pragma unroll
  for (int nd = 0; nd < 2 * KS; ++nd) o[nd][0] = o[nd][1] = o[nd][2] = o[nd][3] = 0.f;

  if (c_begin < c_end) { look_up(c_begin); if (c_begin + 1 < c_end) look_up(c_begin + 1); }
  __syncthreads();
  if (c_begin < c_end) stage(c_begin, 0);
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

  if (NP == 1 && NS == 1) {
#pragma unroll
    for (int hr = 0; hr < 2; ++hr) {
      if (hr ? on_b : on_a) {
        const int q = hr ? qb : qa;
        const float l = hr ? l_b : l_a, inv = l > 0.f ? 1.0f / l : 0.f;
        bf16* orow = P.o + (size_t)(off + q / G) * nq + (size_t)(kvh * G + q % G) * hd + t4 * 2;
#pragma unroll
        for (int nd = 0; nd < 2 * KS; ++nd)
          if (EXACT || nd < ntiles) {
            const float v0 = o[nd][2 * hr] * inv, v1 = o[nd][2 * hr + 1] * inv;
            const __nv_bfloat162 h2 = __floats2bfloat162_rn(v0, v1);
            *reinterpret_cast<__nv_bfloat162*>(orow + nd * 8) = h2;
            *reinterpret_cast<uint32_t*>(orow + (size_t)P.lo_row * nq + nd * 8) = mk::pack_bf16x2(v0 - __low2float(h2), v1 - __high2float(h2));
          }
      }
    }
    return;
  }
  // states [part][query][hd + 4] (O, then max and sum) in the staging area, merged over parts and ranges
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

// Embedding of the pass's rows (tok, pos, req written by k_rows): the residual stream, the first GEMM's
// operand bf16(x * gain) hi + lo, the row's statistics, its rotation table and its cache row.  One block per row.
__global__ void __launch_bounds__(256) k_wide_embed(const bf16* __restrict__ tok_emb, const bf16* __restrict__ pos_emb, const int* __restrict__ tok,
                                                    const int* __restrict__ pos, const int* __restrict__ req, const int* __restrict__ page_table,
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
