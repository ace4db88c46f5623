// GEMMs of passes over 65 to 128 rows (serving batches, short prompts).  At these sizes a pass is bound by the weights, like the
// persistent kernel's, but has one row tile only: with the rows on the MMA's M side (wide.cuh) a launch is as many
// column tiles as CTAs can be fed with, each a long chain of k-blocks of eight MMAs, and two thirds of the loads are rows that
// every CTA reads again.  Here the weights are the M side (128 features or whole heads per CTA, two CTAs to an MMA: cta_group::2)
// and the rows the N side: the even CTA holds their hi parts, the odd one their lo parts, and one MMA of N = 2 x rows covers both.
//
// A cluster of C pairs shares a pair of tiles: every pair multiplies a range of K, every CTA puts its partial tile (rows x 128, fp32) into its
// shared memory and finishes an equal share of the rows, whose partial sums it reads from the cluster's CTAs in K order.  So the few tiles of a narrow GEMM still
// use the chip, the sums cross a cluster and not the L2, and the epilogue's work is spread evenly.  (A cluster's CTAs run together
// by construction; CTAs that wait for each other through global memory would need a cooperative launch.)
//
// Bound by what an SM takes in: a k-block (16 KB of weights, 14 KB of rows, 112 rows) takes 0.34 us, 88 KB a us, of 105 at most;
// then the epilogue (1 us to move the sums to shared memory, 2.4 to 4.7 us) and the hand-over to the next launch (2 to 3 us), both exposed.
// Validate calls, before and after: 3B, 97 rows of 16 requests 4068 -> 2751 us; 0.4B, the same requests 1879 -> 1322; 7B 5506 -> 4362;
// 66 to 128 rows of prefixes of 64 and 400 on all three: 15 to 38 % less.  Tried: single CTAs with all rows each (42 KB a k-block, 0.45 us:
// 3551 us), sums sent to the finishing CTA with four-byte stores (5.5 us a tile: 3878), the exchange tile beside the ring (3211).
//
// Warp roles as in k_wide_gemm (352 threads): warps 0 and 10 TMA producers of weights and rows, warp 1 MMA issuer, warps 2-9 epilogue.
#pragma once
#include "wide.cuh"

namespace stairs {
namespace mid {

using namespace tc;
using mk::store_split4;
using mk::pack_f16x2;
using wide::WideJob;

constexpr int M_MAX_ROWS = 128;
constexpr int X_LD = 132;                  // row pitch (floats) of the exchange tile
constexpr int MAX_C = 4;                   // pairs of a cluster

__device__ __forceinline__ bool mbar_try_cluster(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.b32 %0, 1, 0, p;\n\t}"
      : "=r"(ok) : "r"(smem_u32(bar)), "r"(parity) : "memory");
  return ok != 0;
}
__device__ __forceinline__ bool mbar_wait_cluster(uint64_t* bar, uint32_t parity, volatile int* abort_flag, unsigned long long limit) {
  if (mbar_try_cluster(bar, parity)) return true;
  const long long t0 = clock64();
  while (true) {
    if (mbar_try_cluster(bar, parity)) return true;
    if (*abort_flag) return false;
    if ((unsigned long long)(clock64() - t0) > limit) { *abort_flag = 1; return false; }
  }
}
__device__ __forceinline__ void mbar_arrive_rank(uint64_t* bar, uint32_t rank) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(wide::map_rank(smem_u32(bar), rank)) : "memory");
}

__device__ __forceinline__ void commit_pair(uint64_t* bar, uint16_t mask) {   // arrives on both CTAs' copies of the barrier
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
               ::"r"(smem_u32(bar)), "h"(mask) : "memory");
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }

__device__ __forceinline__ void tmem_ld16_issue(uint32_t taddr, uint32_t* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr) : "memory");
}

// Does every cluster of the launch have one pair of tiles at most?
__host__ __device__ inline bool one_round(const WideJob& job, int grid) { return (job.n_tiles + 1) / 2 * 2 * job.splits <= grid; }

// SPLIT: K is cut over several pairs (C > 1).
template <int EPI, bool SPLIT>
__global__ void __launch_bounds__(wide::WTHREADS, 1) k_mid_gemm(const __grid_constant__ WideJob job) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  const int TN = job.TN, stages = job.stages, C = SPLIT ? job.splits : 1, T = job.T, xb = job.x_box;
  const int w_bytes = TN * BK * 2, stage_bytes = w_bytes + xb * BK * 2;
  uint8_t* tail = smem + (size_t)stages * stage_bytes;
  // [T][X_LD] this CTA's partial tile: in the ring where the CTA has one tile only (its loads and MMAs are over by then), else behind it
  const bool alone = one_round(job, gridDim.x);
  float* xch = reinterpret_cast<float*>(alone ? smem : tail);
  float* rstd = reinterpret_cast<float*>(alone ? tail : tail + (size_t)xb * X_LD * 4);                   // [128] row statistics (of this CTA's rows)
  float* mean = rstd + M_MAX_ROWS;
  float* colc = mean + M_MAX_ROWS;                                   // [2][u, c, gain][128] of the tile's columns
  uint64_t* full = reinterpret_cast<uint64_t*>(colc + 2 * 3 * 128);
  uint64_t* empty = full + wide::W_MAX_STAGES;
  uint64_t* acc_full = empty + wide::W_MAX_STAGES;                   // [2]
  uint64_t* acc_empty = acc_full + 2;                                // [2]
  uint64_t* x_full = acc_empty + 2;                                  // the exchange tiles of all K ranges are complete
  uint64_t* x_empty = x_full + 1;                                    // ... and all have read their share of this CTA's
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(x_empty + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = (int)wide::cluster_rank(), z = rank >> 1, h = rank & 1;   // K range, half of the pair
  const int cid = blockIdx.x / (2 * C), n_cl = gridDim.x / (2 * C), n_pairs = (job.n_tiles + 1) / 2;
  const int kb0 = job.kblocks * z / C, kb1 = job.kblocks * (z + 1) / C;
  uint32_t tmem_cols = 32;
  while ((int)tmem_cols < 4 * xb) tmem_cols <<= 1;

  if (threadIdx.x == 0) {
    for (int s = 0; s < stages; ++s) { mbar_init(full + s, 1); mbar_init(empty + s, 1); }
    mbar_init(acc_full + 0, 1); mbar_init(acc_full + 1, 1);
    mbar_init(acc_empty + 0, 2 * wide::EPI_WARPS); mbar_init(acc_empty + 1, 2 * wide::EPI_WARPS);
    mbar_init(x_full, wide::EPI_WARPS * C); mbar_init(x_empty, wide::EPI_WARPS * C);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) wide::w_alloc<2>(tmem_slot, tmem_cols);
  tc_fence_before();
  __syncthreads();
  wide::cluster_sync();                    // the other CTAs' barriers are ready to be arrived on
  tc_fence_after();
  __syncthreads();
  const uint32_t tmem_base = *tmem_slot;
  if (threadIdx.x == 0) wide::pdl_launch();   // (after the TMEM allocation, see k_wide_attn_tc)
  int issued = 0, p_stage = 0;
  uint32_t p_phase = 0;
  bool arrived = false;                    // on the cluster barrier that ends the kernel

  if (warp == 0) {
    // ------------------------------------------------------------------ TMA producer, weight tiles (they depend on nothing)
    if (lane == 0) {
      const uint64_t pol_w = policy_evict_first();
      int stage = 0; uint32_t phase = 0;
      bool ok = true;
      for (int pt = cid; pt < n_pairs && ok; pt += n_cl) {
        int src = 0, local = 2 * pt + h;      // (past the last tile of an odd number: rows past the matrix, zeros)
        while (src + 1 < job.n_src && local >= job.src_tiles[src]) { local -= job.src_tiles[src]; ++src; }
        for (int kb = kb0; kb < kb1; ++kb) {
          if (!mbar_wait(empty + stage, phase ^ 1, abort_flag, job.wait_limit)) { ok = false; break; }
          if (h == 0) mbar_expect_tx(full + stage, (uint32_t)(2 * stage_bytes));   // (both CTAs' copies)
          wide::w_tma<2>(smem + (size_t)stage * stage_bytes, &job.w_map[src], kb * BK, local * TN, full + stage, pol_w);
          ++issued;
          if (++stage == stages) { stage = 0; phase ^= 1; }
          p_stage = stage; p_phase = phase;
        }
      }
    }
  } else if (warp == 10) {
    // ------------------------------------------------------------------ TMA producer, rows
    if (lane == 0) {
      const uint64_t pol_x = policy_evict_last();
      wide::pdl_wait();
      int stage = 0; uint32_t phase = 0;
      bool ok = true;
      for (int pt = cid; pt < n_pairs && ok; pt += n_cl)
        for (int kb = kb0; kb < kb1; ++kb) {
          if (!mbar_wait(empty + stage, phase ^ 1, abort_flag, job.wait_limit)) { ok = false; break; }
          wide::w_tma3<2>(smem + (size_t)stage * stage_bytes + w_bytes, &job.x_map, kb * BK, 0, h, full + stage, pol_x);   // hi or lo rows
          if (++stage == stages) { stage = 0; phase ^= 1; }
        }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer (the pair's even CTA)
    if (lane == 0 && h == 0) {
      const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)((2 * xb) >> 3) << 17) | ((uint32_t)(256 >> 4) << 24);   // M = 256, N = 2 xb
      const uint16_t pair = (uint16_t)(3u << rank);
      int stage = 0; uint32_t phase = 0;
      int buf = 0; uint32_t acc_bits = 0;
      bool ok = true;
      for (int pt = cid; pt < n_pairs && ok; pt += n_cl) {
        if (!mbar_wait(acc_empty + buf, ((acc_bits >> buf) & 1u) ^ 1u, abort_flag, job.wait_limit)) break;
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + (uint32_t)buf * (tmem_cols / 2);
        for (int kb = kb0; kb < kb1; ++kb) {
          if (!mbar_wait(full + stage, phase, abort_flag, job.wait_limit)) { ok = false; break; }
          tc_fence_after();
          // (a weight tile of fewer than 128 rows: the MMA's other lanes multiply whatever follows it, and nobody reads them)
          const uint32_t a = smem_u32(smem + (size_t)stage * stage_bytes);
          const uint64_t w = smem_desc_sw128(a), x = smem_desc_sw128(a + w_bytes);
#pragma unroll
          for (int k = 0; k < BK / UMMA_K; ++k)
            wide::w_mma<2>(d_tmem, w + (uint64_t)(k * UMMA_K * 2 / 16), x + (uint64_t)(k * UMMA_K * 2 / 16), idesc, (kb > kb0 || k > 0) ? 1u : 0u);
          commit_pair(empty + stage, pair);
          if (++stage == stages) { stage = 0; phase ^= 1; }
        }
        if (!ok) break;
        commit_pair(acc_full + buf, pair);
        acc_bits ^= 1u << buf; buf ^= 1;
      }
    }
  } else {
    // ------------------------------------------------------------------ epilogue (warps 2..9)
    const int quad = warp & 3, hw = (warp - 2) >> 2, et = threadIdx.x - 64;
    const int er = et >> 3, cg = et & 7;               // row of a pass of 32 rows, column groups of the thread
    const int r_begin = T * z / C, r_end = T * (z + 1) / C;
    wide::pdl_wait();
    if (job.norm_in) {
      // row statistics of this CTA's rows, eight lanes per row: merged count-weighted mean, then M2
      const int sub = lane & 7;
      for (int r0 = r_begin; r0 < r_end; r0 += 32) {
        const int r = r0 + er;
        const float4* sr = job.stats_in + (size_t)min(r, r_end - 1) * job.stat_tiles_in;
        float n = 0.f, s1 = 0.f, s2 = 0.f, m0 = 0.f;     // (sums shifted by the lane's first mean)
        for (int i0 = sub; i0 < job.stat_tiles_in; i0 += 32) {
          float4 e[4];
#pragma unroll
          for (int i = 0; i < 4; ++i) e[i] = i0 + 8 * i < job.stat_tiles_in ? __ldcg(sr + i0 + 8 * i) : make_float4(0.f, 0.f, 0.f, 0.f);
          if (i0 == sub) m0 = e[0].x;
#pragma unroll
          for (int i = 0; i < 4; ++i) { const float d0 = e[i].x - m0, nd = e[i].z * d0; n += e[i].z; s1 += nd; s2 += e[i].y + nd * d0; }
        }
        const float mean_l = m0 + s1 / fmaxf(n, 1.f), m2_l = fmaxf(s2 - s1 * s1 / fmaxf(n, 1.f), 0.f);
        float n_all = n, w = n * mean_l;
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) { n_all += __shfl_xor_sync(0xffffffffu, n_all, o); w += __shfl_xor_sync(0xffffffffu, w, o); }
        const float m = w / fmaxf(n_all, 1.f);
        float m2 = m2_l + n * (mean_l - m) * (mean_l - m);
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) m2 += __shfl_xor_sync(0xffffffffu, m2, o);
        if (sub == 0 && r < r_end) {
          if (job.norm_kind == 0) { mean[r] = m; rstd[r] = 1.0f / sqrtf(m2 / (float)job.d + job.eps); }
          else { mean[r] = 0.f; rstd[r] = 1.0f / sqrtf((m2 + n_all * m * m) / (float)job.d + job.eps); }
        }
      }
      wide::group_sync();
    }
    int buf = 0; uint32_t acc_bits = 0, x_par = 0, n_done = 0;
    bool first = true, ok = true;
    for (int pt = cid; pt < n_pairs && ok; pt += n_cl) {
      const int tile = 2 * pt + h;
      int src = 0, local = tile;
      while (src + 1 < job.n_src && local >= job.src_tiles[src]) { local -= job.src_tiles[src]; ++src; }
      const int part = src + job.src0;
      const int n0 = local * TN;                       // first weight row of the tile in its source
      const int ncols = tile >= job.n_tiles ? 0 : EPI == wide::W_SWIGLU ? 64 : min(TN, job.src_rows[src] - n0);
      // The thread's four column groups of four.  QKV: two rotation pairs (a group of a head's first half and its partner
      // half a head further); gate and up tiles: two gate groups and the matching up groups 64 further.
      int col[4];
      bool con[4];
      const int half = job.hd / 2;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        if (EPI == wide::W_QKV) {
          const int pair = cg + 8 * (q >> 1), per = job.hd / 8;   // pairs of groups per head
          const int head = pair / per, i = (pair % per) * 4;
          col[q] = head * job.hd + i + (q & 1) * half;
          con[q] = head * job.hd + job.hd <= ncols;
          if (!con[q]) col[q] = 0;                     // (its values go nowhere)
        } else if (EPI == wide::W_SWIGLU) { col[q] = (cg + 8 * (q >> 1)) * 4 + (q & 1) * 64; con[q] = ncols > 0; }
        else { col[q] = (cg + 8 * q) * 4; con[q] = col[q] < ncols; }
      }
      // per-column constants of the tile: folded LayerNorm's u and c, the next operand's gain.  (Two sets: a warp starts a tile only
      // after every warp has finished the one before the last.)
      float* uc = colc + (n_done & 1) * 3 * 128;
      ++n_done;
      if (et < 128) {
        const bool m_on = EPI == wide::W_SWIGLU ? ncols > 0 : et < ncols;
        if (job.norm_in && job.u) {
          const int n = EPI == wide::W_QKV ? job.u_off[src] + n0 + et : EPI == wide::W_SWIGLU ? (et >> 6) * job.N + tile * 64 + (et & 63) : n0 + et;
          uc[et] = m_on ? __ldg(job.u + n) : 0.f;
          uc[128 + et] = m_on ? __ldg(job.c + n) : 0.f;
        }
        if (EPI == wide::W_ADD && job.next_g) uc[256 + et] = m_on ? __ldg(job.next_g + n0 + et) : 0.f;
      }
      // old residual values / rotation table entries and cache row of the thread's rows of the first pass
      constexpr int NR = SPLIT ? 1 : 2;                // rows of a thread in flight together (r and r + 32)
      float4 pre[NR][4];
      int kv_row[NR], tab[2];
      if (EPI == wide::W_QKV) { tab[0] = (cg % (job.hd / 8)) * 4; tab[1] = ((cg + 8) % (job.hd / 8)) * 4; }
      auto fetch_rows = [&](int r0) {
#pragma unroll
        for (int j = 0; j < NR; ++j) {
          const int r = r0 + 32 * j;
          if (EPI == wide::W_ADD) {
#pragma unroll
            for (int q = 0; q < 4; ++q)
              pre[j][q] = r < r_end && con[q] ? __ldcg(reinterpret_cast<const float4*>(job.out_f32 + (size_t)r * job.ldo + n0 + col[q])) : make_float4(0.f, 0.f, 0.f, 0.f);
          } else if (EPI == wide::W_QKV && r < r_end) {
            kv_row[j] = part == 0 ? r : __ldcg(job.kv_row + r);
            if (job.rope && part < 2) {
#pragma unroll
              for (int p = 0; p < 2; ++p) {
                pre[j][2 * p] = __ldcg(reinterpret_cast<const float4*>(job.rope_cs + (size_t)r * half + tab[p]));
                pre[j][2 * p + 1] = __ldcg(reinterpret_cast<const float4*>(job.rope_sn + (size_t)r * half + tab[p]));
              }
            }
          }
        }
      };
      fetch_rows(r_begin + er);
      ok = mbar_wait(acc_full + buf, (acc_bits >> buf) & 1u, abort_flag, job.wait_limit);
      if (ok && !first) ok = mbar_wait_cluster(x_empty, x_par ^ 1u, abort_flag, job.wait_limit);   // the last tile's sums have been read everywhere
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      acc_bits ^= 1u << buf;
      tc_fence_after();
      const uint32_t taddr = tmem_base + ((uint32_t)(quad * 32) << 16) + (uint32_t)buf * (tmem_cols / 2);
#pragma unroll 1
      for (int c0 = hw * 16; c0 < T; c0 += 32) {       // (rolled: code that runs once costs its fetch)
        uint32_t v[32];
        tmem_ld16_issue(taddr + (uint32_t)c0, v);
        tmem_ld16_issue(taddr + (uint32_t)(xb + c0), v + 16);
        wide::tmem_ld_wait<32>(v);
        float* o = xch + (size_t)c0 * X_LD + quad * 32 + lane;   // (rows past T: the tile has x_box of them)
#pragma unroll
        for (int j = 0; j < 16; ++j) o[j * X_LD] = __uint_as_float(v[j]) + __uint_as_float(v[16 + j]);
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_rank(acc_empty + buf, rank & ~1);
      if (lane < C) mbar_arrive_rank(x_full, 2 * lane + h);
      buf ^= 1;
      ok = __all_sync(0xffffffffu, mbar_wait_cluster(x_full, x_par, abort_flag, job.wait_limit));
      if (!ok) break;
      x_par ^= 1u; first = false;
      for (int rb = r_begin; rb < r_end; rb += 32 * NR) {
        float4 a[NR][4];
        const int ra = rb + er;
#pragma unroll
        for (int j = 0; j < NR; ++j) {
          const int r = ra + 32 * j;
#pragma unroll
          for (int q = 0; q < 4; ++q) a[j][q] = make_float4(0.f, 0.f, 0.f, 0.f);
          if (r < r_end) {
            if (!SPLIT) {
#pragma unroll
              for (int q = 0; q < 4; ++q) a[j][q] = *reinterpret_cast<const float4*>(xch + (size_t)r * X_LD + col[q]);
            } else {
              const uint32_t at = smem_u32(xch + (size_t)r * X_LD);
              float4 p[MAX_C][4];                      // (every load in flight: another CTA's memory is a long way off)
#pragma unroll
              for (int zz = 0; zz < MAX_C; ++zz) {
                const uint32_t from = wide::map_rank(at, 2 * (zz < C ? zz : z) + h);
#pragma unroll
                for (int q = 0; q < 4; ++q)
                  if (zz < C) p[zz][q] = wide::ld_cluster_f4(from + (uint32_t)col[q] * 4);
              }
#pragma unroll
              for (int zz = 0; zz < MAX_C; ++zz)
#pragma unroll
                for (int q = 0; q < 4; ++q)
                  if (zz < C) { a[j][q].x += p[zz][q].x; a[j][q].y += p[zz][q].y; a[j][q].z += p[zz][q].z; a[j][q].w += p[zz][q].w; }
            }
            if (job.norm_in) {
              const float rs = rstd[r], mu = mean[r];
#pragma unroll
              for (int q = 0; q < 4; ++q) {
                float4& v = a[j][q];
                if (job.u) {
                  const float4 u4 = *reinterpret_cast<const float4*>(uc + col[q]), c4 = *reinterpret_cast<const float4*>(uc + 128 + col[q]);
                  v.x = rs * (v.x - mu * u4.x) + c4.x; v.y = rs * (v.y - mu * u4.y) + c4.y;
                  v.z = rs * (v.z - mu * u4.z) + c4.z; v.w = rs * (v.w - mu * u4.w) + c4.w;
                } else { v.x *= rs; v.y *= rs; v.z *= rs; v.w *= rs; }
              }
            }
          }
        }
        if (rb + 32 * NR >= r_end) {                   // this warp has read its rows: the exchange tiles may be written again
          __syncwarp();
          if (lane < C) mbar_arrive_rank(x_empty, 2 * lane + h);
          if (pt + n_cl >= n_pairs) { cluster_arrive(); arrived = true; }   // (and nothing of this warp's touches another CTA any more)
        }
        if (EPI == wide::W_ADD) {
#pragma unroll
          for (int j = 0; j < NR; ++j)
#pragma unroll
            for (int q = 0; q < 4; ++q) { float4& v = a[j][q]; v = make_float4(pre[j][q].x + v.x, pre[j][q].y + v.y, pre[j][q].z + v.z, pre[j][q].w + v.w); }
          if (rb + 32 * NR < r_end) fetch_rows(ra + 32 * NR);
        }
#pragma unroll
        for (int j = 0; j < NR; ++j) {
          const int r = ra + 32 * j;
          const bool on = r < r_end;
          if (EPI == wide::W_ADD) {
            float s = 0.f, cnt = 0.f;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              const float4 v = a[j][q];
              if (on && con[q]) {
                *reinterpret_cast<float4*>(job.out_f32 + (size_t)r * job.ldo + n0 + col[q]) = v;
                if (job.next_g) {
                  const float4 g4 = *reinterpret_cast<const float4*>(uc + 256 + col[q]);
                  store_split4(job.out_act, (size_t)r * job.ldo + n0 + col[q], (size_t)job.lo_row * job.ldo, make_float4(v.x * g4.x, v.y * g4.y, v.z * g4.z, v.w * g4.w));
                }
                cnt += 4.f; s += (v.x + v.y) + (v.z + v.w);
              }
            }
            if (job.next_g) {
              // the row's statistics over this tile (count, mean, centred sum of squares), by its eight threads
#pragma unroll
              for (int o = 1; o < 8; o <<= 1) { cnt += __shfl_xor_sync(0xffffffffu, cnt, o); s += __shfl_xor_sync(0xffffffffu, s, o); }
              const float m = cnt > 0.f ? s / cnt : 0.f;
              float m2 = 0.f;
#pragma unroll
              for (int q = 0; q < 4; ++q)
                if (con[q]) { const float4 v = a[j][q]; const float d0 = v.x - m, d1 = v.y - m, d2 = v.z - m, d3 = v.w - m; m2 += (d0 * d0 + d1 * d1) + (d2 * d2 + d3 * d3); }
#pragma unroll
              for (int o = 1; o < 8; o <<= 1) m2 += __shfl_xor_sync(0xffffffffu, m2, o);
              if (on && cg == 0 && ncols > 0) job.stats_out[(size_t)r * job.n_tiles + tile] = make_float4(m, m2, cnt, 0.f);
            }
          } else if (EPI == wide::W_GELU) {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              const float2 lo = wide::gelu_erfc2(make_float2(a[j][q].x, a[j][q].y)), hi = wide::gelu_erfc2(make_float2(a[j][q].z, a[j][q].w));
              if (on && con[q]) store_split4(job.out_act, (size_t)r * job.ldo + n0 + col[q], (size_t)job.lo_row * job.ldo, make_float4(lo.x, lo.y, hi.x, hi.y));
            }
          } else if (EPI == wide::W_SWIGLU) {
#pragma unroll
            for (int p = 0; p < 2; ++p) {
              const float4 g = a[j][2 * p], w = a[j][2 * p + 1];
              const float4 v = make_float4(silu_f(g.x) * w.x, silu_f(g.y) * w.y, silu_f(g.z) * w.z, silu_f(g.w) * w.w);
              if (on && con[2 * p]) store_split4(job.out_act, (size_t)r * job.ldo + tile * 64 + col[2 * p], (size_t)job.lo_row * job.ldo, v);
            }
          } else if (EPI == wide::W_LMHEAD) {
            unsigned long long key = 0ull;
            const bool vec = ((job.ldo & 3) | (int)(reinterpret_cast<uintptr_t>(job.out_f32) & 15)) == 0;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              const float e4[4] = {a[j][q].x, a[j][q].y, a[j][q].z, a[j][q].w};
              float* lg = job.out_f32 ? job.out_f32 + (size_t)r * job.ldo + n0 + col[q] : nullptr;
              const bool whole = vec && col[q] + 4 <= ncols;
              if (on && lg && whole) *reinterpret_cast<float4*>(lg) = a[j][q];
#pragma unroll
              for (int e = 0; e < 4; ++e)
                if (on && col[q] + e < ncols) {
                  if (lg && !whole) lg[e] = e4[e];
                  const unsigned long long k2 = argmax_key(e4[e], (uint32_t)(n0 + col[q] + e));
                  key = k2 > key ? k2 : key;
                }
            }
#pragma unroll
            for (int o = 1; o < 8; o <<= 1) { const unsigned long long other = __shfl_xor_sync(0xffffffffu, key, o); key = other > key ? other : key; }
            if (on && cg == 0 && key) atomicMax(job.keys + r, key);
          } else {   // W_QKV: rotate and scale q, rotate k; fp16 to the query buffer and the cache
            const float qs = part == 0 ? job.qscale : 1.0f;
            __half* dst = (part == 0 ? job.q16 : part == 1 ? job.kc : job.vc) + (size_t)(on ? kv_row[j] : 0) * job.src_rows[src] + n0;
#pragma unroll
            for (int p = 0; p < 2; ++p) {
              float4 lo = a[j][2 * p], hi = a[j][2 * p + 1];
              if (job.rope && part < 2) {
                const float4 cs = pre[j][2 * p], sn = pre[j][2 * p + 1], l = lo, g = hi;
                lo = make_float4(l.x * cs.x - g.x * sn.x, l.y * cs.y - g.y * sn.y, l.z * cs.z - g.z * sn.z, l.w * cs.w - g.w * sn.w);
                hi = make_float4(g.x * cs.x + l.x * sn.x, g.y * cs.y + l.y * sn.y, g.z * cs.z + l.z * sn.z, g.w * cs.w + l.w * sn.w);
              }
              if (on && con[2 * p]) {
                *reinterpret_cast<uint2*>(dst + col[2 * p]) = make_uint2(pack_f16x2(lo.x * qs, lo.y * qs), pack_f16x2(lo.z * qs, lo.w * qs));
                *reinterpret_cast<uint2*>(dst + col[2 * p + 1]) = make_uint2(pack_f16x2(hi.x * qs, hi.y * qs), pack_f16x2(hi.z * qs, hi.w * qs));
              }
            }
          }
        }
        if (EPI == wide::W_QKV && rb + 32 * NR < r_end) fetch_rows(ra + 32 * NR);
      }
      if (r_begin >= r_end) {
        __syncwarp();
        if (lane < C) mbar_arrive_rank(x_empty, 2 * lane + h);
      }
    }
  }

  // ------------------------------------------------------------------ teardown
  tc_fence_before();
  __syncthreads();
  if (*abort_flag) {
    if (threadIdx.x == 0) {
      *reinterpret_cast<volatile unsigned int*>(job.status + STATUS_ERROR) = 5u;  // STAIRS_ETIMEOUT
      __threadfence_system();
      // copies in flight must land before the shared memory is given back (bounded).  A pair's copies all signal on the even CTA, so the
      // odd one waits out the bound.
      const long long t0 = clock64();
      const unsigned long long lim = job.wait_limit > 2000000ull ? job.wait_limit : 2000000ull;
      int s = p_stage; uint32_t ph = p_phase;
      for (int i = 0; i < stages && i < issued; ++i) {
        if (--s < 0) { s = stages - 1; ph ^= 1; }
        while (h != 0 || !mbar_try(full + s, ph)) {
          if ((unsigned long long)(clock64() - t0) > lim) break;
        }
      }
      settle(t0);
    }
    __syncthreads();
  }
  if (!arrived) cluster_arrive();
  cluster_wait();                          // no CTA leaves while another may still use its shared memory or barriers
  if (warp == 1) { tc_fence_after(); wide::w_dealloc<2>(tmem_base, tmem_cols); }
}

// x_box: the call's rows, a multiple of 16 (N = 2 x_box has to be one of 32)
inline size_t gemm_smem(int x_box, int TN, int stages, bool alone) {
  const size_t ring = (size_t)stages * (TN + x_box) * BK * 2, xch = (size_t)x_box * X_LD * 4;
  return 1024 + (alone ? std::max(ring, xch) : ring + xch) + (2 * M_MAX_ROWS + 2 * 3 * 128) * 4 + (2 * wide::W_MAX_STAGES + 6) * 8 + 64;
}
inline int gemm_stages(int x_box, int TN, bool alone) {
  int s = wide::W_MAX_STAGES;
  while (s > 3 && gemm_smem(x_box, TN, s, alone) > (size_t)SMEM_LIMIT) --s;
  return s;
}

}  // namespace mid
}  // namespace stairs
