// Whole passes of small fp32 models in one launch of one thread-block cluster.
//
// A pass of such a model (config 1: four layers of width 256, 12 MB of weights) is a chain of dependent steps
// of a microsecond each; launched one by one they cost 4 us apiece (about 45 launches a validate call).  Here
// a cluster of up to 16 CTAs walks the chain with cluster barriers: QKV (feature pairs rotated and filed by
// the same warp), attention, O projection, MLP up, MLP down, at the end the LM head with its argmax and the
// accept step; an assistant's whole draft (k steps) is one launch.  What bounds it is the number of trips to L2 in
// a step, so
//  * activations never leave shared memory: every CTA keeps the residual stream, queries, attention output and
//    MLP activation of the pass's rows, and whoever computes a value stores it into all CTAs' copies (through
//    L2 a step took 5 us, the trip of the residual, of the operand and of the barrier's release);
//  * a warp's weight rows come through a small shared-memory ring; one lane asks for the next step's rows, one bulk
//    copy an item, before it leaves the step (per-lane asynchronous copies took a fifth of a pass to issue);
//  * an attention warp asks for its keys and values at once;
//  * the steps share ONE copy of the code, straight lines with whole batches of loads first.  A step runs a few
//    hundred instructions once per warp, and code that is not in the innermost caches runs at 0.15 instructions a
//    cycle: with the GEMM code instantiated per step 2 us of a step's 5 were the 300 instructions of one dot product.
// Measured (four layers of width 256, 31-token prompt, 64 tokens generated): a validate pass of five rows 105 us (launch
// by launch 220), the draft of four tokens 130 us (330), the whole call 7.24 ms -> 3.41 ms.  What is left is
// latency: about 2.5 us for each of a layer's five steps (barrier and publication 1 us, the rest code that runs once).
// Rows are taken eight at a time (a pass per block of rows: later rows only need earlier rows' K/V); the requests of a
// validate call are dealt to several clusters, which have nothing to do with one another (8 CTAs each where not all of 16 would run at once).
//
// A warp owns whole features; its lanes stride the K dimension in 16-byte vectors and hold one sum per
// (feature, row).  The order of the additions depends on K only, and a row's attention on its position
// only, so results do not depend on the call's other rows.
#pragma once
#include <type_traits>

#include "kernels_basic.cuh"
#include "gemm_simt.cuh"
#include "gemm_tc.cuh"

namespace stairs {
namespace small {

constexpr int S_WARPS = 8, S_THREADS = S_WARPS * 32;
constexpr int S_BLOCK = 8;           // rows of a pass
// Most passes of a launch; whether a call's are quicker than one launch per operation is small_pays' to say.
constexpr int S_MOST_PASSES = 2;
constexpr int S_MAX_HD = 128, S_MAX_REQ = 64, S_MAX_LAYERS = 32, S_MAX_CTAS = 16;
constexpr int S_MAX_CLUSTERS = 8;    // clusters of a validate call, each with requests of its own
constexpr int S_ROWS = S_MAX_CLUSTERS * S_MOST_PASSES * S_BLOCK;   // rows of a call
constexpr int S_GROUP = 4;           // warps that share one (row, head) of the attention
constexpr int S_RING = 16384;        // bytes of a warp's weight ring
constexpr int S_SLOTS = 3;           // items a warp's ring holds at most
constexpr int S_MAP = 8;             // QKV items of a warp whose place is looked up

struct SmallLayer {
  const float *n1w, *n1b, *wq, *wk, *wv, *wo, *n2w, *n2b, *w1, *w3, *w2;
  float *kc, *vc;
};

struct SmallParams {
  const SmallLayer* layers; int n_layers;
  int d, Hq, Hkv, hd, F, vocab, norm_kind, act, rope; float theta, eps;
  const float *tok_emb, *pos_emb, *fnw, *fnb, *head;
  int mode;                          // RowMode; ROWS_DRAFT_FIRST: `steps` assistant steps
  int T, steps, n_req, slot, first, head_rows;   // head_rows 0: no logits (prefill)
  int val_req[S_MAX_REQ], val_k[S_MAX_REQ], val_off[S_MAX_REQ];
  int cl_req[S_MAX_CLUSTERS + 1];    // validate: first request of every cluster, then n_req
  const int* draft; int* draft_out; int k_max;
  int* seq; int* n_seq; int max_seq_len;
  const int* page_table; int page_tokens, max_pages;
  float* logits;
  int* target_tokens; int* accept_len; int commit;
  unsigned int* status; unsigned long long wait_limit;
};

struct SmallSmem {
  int tok[S_BLOCK], pos[S_BLOCK], slot[S_BLOCK], kv[S_BLOCK];
  int result[S_MOST_PASSES * S_BLOCK];                   // argmax of every row of the cluster
  unsigned long long keys[S_BLOCK][S_MAX_CTAS * S_WARPS];  // LM head: every warp's best of every row
  float part[S_WARPS][S_MAX_HD + 4];                     // attention: one warp's output, maximum and sum
  unsigned long long landed[S_WARPS][S_SLOTS];           // mbarriers of the weight rings
  int abort;                                             // a wait ran out: the launch's results are void, its other waits give up at once
  SmallLayer layers[S_MAX_LAYERS];
  int qkv_row[S_WARPS][S_MAP];                           // QKV: matrix (top bits) and first row of a warp's first items
};
// dynamic shared memory: SmallSmem, the warps' weight rings, then x, normed rows, q, o (d or nq wide) and ff, eight rows each
inline size_t smem_bytes(int d, int nq, int F) {
  return ((sizeof(SmallSmem) + 15) & ~(size_t)15) + (size_t)S_WARPS * S_RING + (size_t)S_BLOCK * 4 * (2 * d + 2 * nq + F);
}

__device__ __forceinline__ void cl_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cl_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ uint32_t sm_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
// Stores into every CTA's copy.  The four lanes of a row (lane / 8 = 0..3) hold the same values and take every fourth CTA.
__device__ __forceinline__ void to_all4(float* p, float4 v, int NC, int first) {
  const uint32_t a = sm_addr(p);
#pragma unroll 1
  for (int r = first; r < NC; r += 4)
    asm volatile("{\n\t.reg .b32 t;\n\tmapa.shared::cluster.u32 t, %0, %1;\n\tst.shared::cluster.v4.f32 [t], {%2, %3, %4, %5};\n\t}" ::"r"(a), "r"(r), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
}
__device__ __forceinline__ void to_all2(float* p, float x, float y, int NC, int first) {
  const uint32_t a = sm_addr(p);
#pragma unroll 1
  for (int r = first; r < NC; r += 4)
    asm volatile("{\n\t.reg .b32 t;\n\tmapa.shared::cluster.u32 t, %0, %1;\n\tst.shared::cluster.v2.f32 [t], {%2, %3};\n\t}" ::"r"(a), "r"(r), "f"(x), "f"(y) : "memory");
}
__device__ __forceinline__ void to_all(unsigned long long* p, unsigned long long v, int NC, int first) {
  const uint32_t a = sm_addr(p);
#pragma unroll 1
  for (int r = first; r < NC; r += 4)
    asm volatile("{\n\t.reg .b32 t;\n\tmapa.shared::cluster.u32 t, %0, %1;\n\tst.shared::cluster.u64 [t], %2;\n\t}" ::"r"(a), "r"(r), "l"(v) : "memory");
}
__device__ __forceinline__ void ring_copy(float* dst, const float* src, uint32_t bytes, unsigned long long* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(sm_addr(dst)), "l"(src), "r"(bytes), "r"(sm_addr(bar)) : "memory");
}

// Sums N per-lane values across the warp: on return lane l holds the total of a[l % N].
template <int N> __device__ __forceinline__ float multi_sum(float (&a)[N], int lane) {
#pragma unroll
  for (int h = N / 2; h >= 1; h >>= 1) {
    const bool up = (lane & h) != 0;
#pragma unroll
    for (int i = 0; i < h; ++i) {
      const float send = up ? a[i] : a[i + h], keep = up ? a[i + h] : a[i];
      a[i] = keep + __shfl_xor_sync(0xffffffffu, send, h);
    }
  }
  float v = a[0];
#pragma unroll
  for (int o = N; o < 32; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

enum StepKind { ST_QKV = 0, ST_ATTN = 1, ST_O = 2, ST_UP = 3, ST_DOWN = 4, ST_HEAD = 5 };

__global__ void __launch_bounds__(S_THREADS, 1) k_small(const __grid_constant__ SmallParams P) {
  extern __shared__ __align__(16) uint8_t small_raw[];
  SmallSmem& S = *reinterpret_cast<SmallSmem*>(small_raw);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  int cta, NC;
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(cta));
  asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(NC));
  const int gw = cta * S_WARPS + warp, NW = NC * S_WARPS;
  const bool validating = P.mode == ROWS_VALIDATE;
  const int req0 = validating ? P.cl_req[blockIdx.x / NC] : 0, req1 = validating ? P.cl_req[blockIdx.x / NC + 1] : 0;   // this cluster's requests
  const int off0 = validating ? P.val_off[req0] : 0;         // and first row
  const int nw_log = 31 - __clz(NW);         // (the cluster has 4, 8 or 16 CTAs)
  const int d = P.d, hd = P.hd, half = hd / 2, nq = P.Hq * hd, nkv = P.Hkv * hd, G = P.Hq / P.Hkv;
  float* ring = reinterpret_cast<float*>(small_raw + ((sizeof(SmallSmem) + 15) & ~(size_t)15)) + (size_t)warp * (S_RING / 4);
  float* sx = reinterpret_cast<float*>(small_raw + ((sizeof(SmallSmem) + 15) & ~(size_t)15) + (size_t)S_WARPS * S_RING);
  float* sn = sx + (size_t)S_BLOCK * d;      // normalised rows
  float* sq = sn + (size_t)S_BLOCK * d;
  float* so = sq + (size_t)S_BLOCK * nq;
  float* sf = so + (size_t)S_BLOCK * nq;
  const int tl = lane & 7, fl = lane >> 3;   // row and feature of this lane's sum
  const float scale = 1.0f / sqrtf((float)hd);

  for (int i = tid; i < P.n_layers * (int)(sizeof(SmallLayer) / 8); i += S_THREADS)
    reinterpret_cast<unsigned long long*>(S.layers)[i] = reinterpret_cast<const unsigned long long*>(P.layers)[i];
  for (int j = lane; j < S_MAP; j += 32) {
    const int it = gw + j * NW, h = 2 * it / half, i = 2 * it % half, m = h < P.Hq ? 0 : h < P.Hq + P.Hkv ? 1 : 2;
    S.qkv_row[warp][j] = (m << 28) | ((h - (m == 0 ? 0 : m == 1 ? P.Hq : P.Hq + P.Hkv)) * hd + i);
  }
  if (lane < S_SLOTS) tc::mbar_init(reinterpret_cast<uint64_t*>(&S.landed[warp][lane]), 1);
  if (tid == 0) S.abort = 0;
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  __syncthreads();                           // S.layers
  cl_arrive();
  cl_wait();                                 // every CTA runs: its shared memory may be written

  unsigned phases = 0, flying = 0;           // ring slots: parity of the next wait, copies not yet waited for
  int T = 0, rows = 0;                       // rows of this step, of this pass
  for (int step = 0; step < P.steps; ++step) {
    T = P.mode == ROWS_DRAFT_FIRST ? (step == 0 ? 2 : 1) : validating ? (req1 < P.n_req ? P.val_off[req1] : P.T) - off0 : P.T;
    for (int r0 = 0; r0 < T; r0 += S_BLOCK) {
      rows = min(S_BLOCK, T - r0);
      // ------------------------------------------------------------ rows of this pass
      if (tid < rows) {
        const int tg = off0 + r0 + tid;
        int token, pos, slot = P.slot;
        if (P.mode == ROWS_VALIDATE) {
          int i = req0;
          while (i + 1 < P.n_req && P.val_off[i + 1] <= tg) ++i;
          slot = P.val_req[i];
          const int base = P.n_seq[slot] - 1, r = tg - P.val_off[i];
          pos = base + r;
          token = r == 0 ? P.seq[(size_t)slot * P.max_seq_len + base] : P.draft[i * P.k_max + r - 1];
        } else if (P.mode == ROWS_PREFILL) {
          pos = P.first + tg;
          token = P.seq[(size_t)slot * P.max_seq_len + pos];
        } else {
          const int n = P.n_seq[slot];
          pos = step == 0 ? n - 2 + tg : n - 1 + step;
          token = step == 0 ? P.seq[(size_t)slot * P.max_seq_len + pos] : S.result[step == 1 ? 1 : 0];
        }
        S.tok[tid] = min(max(token, 0), P.vocab - 1); S.pos[tid] = pos; S.slot[tid] = slot;
        S.kv[tid] = P.page_table[(size_t)slot * P.max_pages + pos / P.page_tokens] * P.page_tokens + pos % P.page_tokens;
      }
      __syncthreads();
      if (warp < rows) {                     // embedding, by every CTA for itself
        const float* e = P.tok_emb + (size_t)S.tok[warp] * d;
        const float* pe = P.pos_emb ? P.pos_emb + (size_t)S.pos[warp] * d : nullptr;
        for (int i = lane * 4; i < d; i += 128) {
          float4 v = __ldg(reinterpret_cast<const float4*>(e + i));
          if (pe) { const float4 p4 = __ldg(reinterpret_cast<const float4*>(pe + i)); v.x += p4.x; v.y += p4.y; v.z += p4.z; v.w += p4.w; }
          *reinterpret_cast<float4*>(sx + (size_t)warp * d + i) = v;
        }
        __syncwarp();
      }
      // four warps per (row, head), 32 positions each at a time
      auto attention = [&](const SmallLayer& L) {
        const int grp = warp / S_GROUP, gwarp = warp % S_GROUP, gt = tid % (S_GROUP * 32), w0 = grp * S_GROUP;
        auto group_sync = [&]() { asm volatile("bar.sync %0, 128;" ::"r"(1 + grp) : "memory"); };
        // A K or V row is read by half a warp (head sizes up to 64) or a whole one, 16 bytes a lane: two rows, or one, per
        // instruction.  (One position per lane touched 32 lines with every load.)  Lane l scores position pos_l.
        const bool two = hd <= 64;
        const int vp = two ? lane >> 4 : 0, vd = (two ? lane & 15 : lane) * 4, chunks = two ? 1 : 2;
        const bool von = vd < hd;
        for (int item = cta * 2 + grp; item < rows * P.Hq; item += NC * 2) {
          const int t = item / P.Hq, h = item - t * P.Hq, kvh = h / G, last = S.pos[t];
          const int* pt = P.page_table + (size_t)S.slot[t] * P.max_pages;
          const float4 q4 = von ? *reinterpret_cast<const float4*>(sq + (size_t)t * nq + (size_t)h * hd + vd) : make_float4(0.f, 0.f, 0.f, 0.f);
          float m = -INFINITY, lsum = 0.f;
          float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);            // this lane's four columns, over its value rows
          for (int base = gwarp * 32; base <= last; base += S_GROUP * 32) {
            const int pos_l = base + (two ? 2 * (lane & 15) + (lane >> 4) : lane), pc = min(base + lane, last), pg = pc / P.page_tokens;
            const int row = __ldg(pt + pg) * P.page_tokens + pc - pg * P.page_tokens;   // of position base + lane
            const size_t head_off = (size_t)kvh * hd + vd;
            float4 va[16];
            float s = -INFINITY;
            for (int c = 0; c < chunks; ++c) {
              float a[16];
              float4 ka[16];
#pragma unroll
              for (int j = 0; j < 16; ++j) {
                const int rj = __shfl_sync(0xffffffffu, row, two ? 2 * j + vp : 16 * c + j);   // (rows past the last position repeat it)
                ka[j] = von ? __ldcg(reinterpret_cast<const float4*>(L.kc + (size_t)rj * nkv + head_off)) : make_float4(0.f, 0.f, 0.f, 0.f);
                if (two) va[j] = von ? __ldcg(reinterpret_cast<const float4*>(L.vc + (size_t)rj * nkv + head_off)) : make_float4(0.f, 0.f, 0.f, 0.f);
              }
#pragma unroll
              for (int j = 0; j < 16; ++j) a[j] = fmaf(ka[j].x, q4.x, fmaf(ka[j].y, q4.y, fmaf(ka[j].z, q4.z, ka[j].w * q4.w)));
#pragma unroll
              for (int hb = 8; hb >= 1; hb >>= 1) {                // sums over 16 lanes: lane l keeps a[l % 16]
                const bool up = (lane & hb) != 0;
#pragma unroll
                for (int i = 0; i < hb; ++i) {
                  const float send = up ? a[i] : a[i + hb], keep = up ? a[i + hb] : a[i];
                  a[i] = keep + __shfl_xor_sync(0xffffffffu, send, hb);
                }
              }
              if (!two) a[0] += __shfl_xor_sync(0xffffffffu, a[0], 16);
              if (two || (lane >> 4) == c) s = a[0];
            }
            if (pos_l > last) s = -INFINITY;
            const float mn = fmaxf(m, warp_max(s));
            const float e = pos_l <= last ? expf(s - mn) : 0.f, corr = expf(m - mn);
            lsum = lsum * corr + warp_sum(e);
            acc.x *= corr; acc.y *= corr; acc.z *= corr; acc.w *= corr;
            m = mn;
            for (int c = 0; c < chunks; ++c) {
              if (!two) {
#pragma unroll
                for (int j = 0; j < 16; ++j) {
                  const int rj = __shfl_sync(0xffffffffu, row, 16 * c + j);
                  va[j] = von ? __ldcg(reinterpret_cast<const float4*>(L.vc + (size_t)rj * nkv + head_off)) : make_float4(0.f, 0.f, 0.f, 0.f);
                }
              }
#pragma unroll
              for (int j = 0; j < 16; ++j) {
                const float ej = __shfl_sync(0xffffffffu, e, two ? 16 * vp + j : 16 * c + j);   // (0 past the last position)
                acc.x = fmaf(ej, va[j].x, acc.x); acc.y = fmaf(ej, va[j].y, acc.y); acc.z = fmaf(ej, va[j].z, acc.z); acc.w = fmaf(ej, va[j].w, acc.w);
              }
            }
          }
          if (two) {   // the two half-warps' value rows
            acc.x += __shfl_xor_sync(0xffffffffu, acc.x, 16); acc.y += __shfl_xor_sync(0xffffffffu, acc.y, 16);
            acc.z += __shfl_xor_sync(0xffffffffu, acc.z, 16); acc.w += __shfl_xor_sync(0xffffffffu, acc.w, 16);
          }
          if (von && vp == 0) *reinterpret_cast<float4*>(&S.part[warp][vd]) = acc;
          if (lane == 0) *reinterpret_cast<float2*>(&S.part[warp][S_MAX_HD]) = make_float2(m, lsum);
          group_sync();
          // the four warps' states; every warp of the group sends the result to a quarter of the CTAs
          const int n_act = min(S_GROUP, last / 32 + 1);           // (the other warps had no positions)
          float M = -INFINITY, Ls = 0.f;
          float2 ml[S_GROUP];
#pragma unroll
          for (int w = 0; w < S_GROUP; ++w) {
            ml[w] = w < n_act ? *reinterpret_cast<const float2*>(&S.part[w0 + w][S_MAX_HD]) : make_float2(-INFINITY, 0.f);
            M = fmaxf(M, ml[w].x);
          }
          float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
          for (int w = 0; w < S_GROUP; ++w)
            if (w < n_act) {
              const float wt = expf(ml[w].x - M);
              Ls += ml[w].y * wt;
              if (lane * 4 < hd) {
                const float4 v = *reinterpret_cast<const float4*>(&S.part[w0 + w][lane * 4]);
                o.x += v.x * wt; o.y += v.y * wt; o.z += v.z * wt; o.w += v.w * wt;
              }
            }
          if (lane * 4 < hd) to_all4(so + (size_t)t * nq + (size_t)h * hd + lane * 4, make_float4(o.x / Ls, o.y / Ls, o.z / Ls, o.w / Ls), NC, gwarp);
          if (item + NC * 2 < rows * P.Hq) group_sync();
        }
      };
      const bool on_row = tl < rows;
      const int n_steps = P.head_rows ? 5 * P.n_layers + 1 : 5 * P.n_layers - 4;   // (a prefill's last layer: its keys and values are all that is read)
      // QKV item: matrix and first row (looked up for a warp's first items: divisions are long code)
      auto qkv_at = [&](int it) {
        const int j = (it - gw) >> nw_log;
        if (j < S_MAP) return S.qkv_row[warp][j];
        const int h = 2 * it / half, i = 2 * it % half, m = h < P.Hq ? 0 : h < P.Hq + P.Hkv ? 1 : 2;
        return (m << 28) | ((h - (m == 0 ? 0 : m == 1 ? P.Hq : P.Hq + P.Hkv)) * hd + i);
      };
      const bool swiglu = P.act == 1;
      auto depth_of = [&](int kind) { return kind == ST_O ? nq : kind == ST_DOWN ? P.F : d; };
      auto items_of = [&](int kind) { return kind == ST_QKV ? (nq + 2 * nkv) / 4 : kind == ST_UP ? P.F / (swiglu ? 2 : 4) : kind == ST_HEAD ? (P.vocab + 3) / 4 : d / 4; };
      // The two pairs of weight rows of an item: QKV: (i, i + 1) and (i + hd/2, i + 1 + hd/2) of a head; SwiGLU: two gate
      // rows and two up rows; else four rows in order.
      auto rows_of = [&](const SmallLayer& L, int kind, int K, int it, const float*& p0, const float*& p1) {
        if (kind == ST_QKV) {
          const int at = qkv_at(it), m = at >> 28;
          p0 = (m == 0 ? L.wq : m == 1 ? L.wk : L.wv) + (size_t)(at & 0x0fffffff) * K;
          p1 = p0 + (size_t)half * K;
        } else if (kind == ST_UP && swiglu) {
          p0 = L.w1 + (size_t)(2 * it) * K; p1 = L.w3 + (size_t)(2 * it) * K;
        } else {
          p0 = (kind == ST_O ? L.wo : kind == ST_DOWN ? L.w2 : kind == ST_HEAD ? P.head : L.w1) + (size_t)(4 * it) * K;
          p1 = p0 + 2 * (size_t)K;
        }
      };
#pragma unroll 1
      for (int st = -1; st < n_steps; ++st) {                         // (-1: only asks for the first step's weights)
        const int l = min(max(st, 0) / 5, P.n_layers - 1), kind = st < 0 ? ST_ATTN : st == 5 * P.n_layers ? ST_HEAD : st % 5;
        const SmallLayer& L = S.layers[l];
        const int K = depth_of(kind), per = 4 * K, slots = min(S_SLOTS, S_RING / 4 / per);   // items the ring holds (0: rows are read from memory)
        const bool gemm = kind != ST_ATTN;
        // the item that goes into a ring slot: one lane asks for it, in one or two bulk copies
        auto fetch = [&](const SmallLayer& Lf, int kf, int Kf, int it, int slot) {
          float* dst = ring + (size_t)slot * 4 * Kf;
          const float *p0, *p1;
          rows_of(Lf, kf, Kf, it, p0, p1);
          const bool split = kf == ST_QKV || (kf == ST_UP && swiglu);
          const uint32_t n = (uint32_t)(kf == ST_HEAD ? min(4, P.vocab - 4 * it) : 4) * (uint32_t)Kf * 4;
          if (*reinterpret_cast<volatile int*>(&S.abort)) return;
          flying |= 1u << slot;
          if (lane == 0) {
            tc::mbar_expect_tx(reinterpret_cast<uint64_t*>(&S.landed[warp][slot]), n);
            ring_copy(dst, p0, split ? n / 2 : n, &S.landed[warp][slot]);
            if (split) ring_copy(dst + 2 * Kf, p1, n / 2, &S.landed[warp][slot]);
          }
        };
        if (st >= 0 && !gemm) {
          cl_wait();
          attention(L);
        }
        if (gemm) {
          // -------------------------------------------------------- a GEMM step: items of four features
          const bool glu = kind == ST_UP && swiglu, pairs = glu || kind == ST_QKV;
          const int items = items_of(kind);
          const float* act = kind == ST_O ? so : kind == ST_DOWN ? sf : sn;
          const float* g = kind == ST_QKV ? L.n1w : kind == ST_UP ? L.n2w : P.fnw;
          const float* b = kind == ST_QKV ? L.n1b : kind == ST_UP ? L.n2b : P.fnb;
          float4 g0 = make_float4(0.f, 0.f, 0.f, 0.f), g1 = g0, b0 = g0, b1 = g0;   // gains and biases of this lane's first two vectors
          if (act == sn && warp < rows) {
            if (lane * 4 < d) { g0 = __ldg(reinterpret_cast<const float4*>(g + lane * 4)); if (b) b0 = __ldg(reinterpret_cast<const float4*>(b + lane * 4)); }
            if (lane * 4 + 128 < d) { g1 = __ldg(reinterpret_cast<const float4*>(g + lane * 4 + 128)); if (b) b1 = __ldg(reinterpret_cast<const float4*>(b + lane * 4 + 128)); }
          }
          cl_wait();                                                   // the step's input is published
          if (act == sn) {
            // one warp per row: normalised x
            if (warp < rows) {
              const float* x = sx + (size_t)warp * d;
              float s = 0.f, ss = 0.f;
#pragma unroll 1
              for (int i = lane * 4; i < d; i += 128) { const float4 v = *reinterpret_cast<const float4*>(x + i); s += (v.x + v.y) + (v.z + v.w); }
              const float mean = P.norm_kind == 0 ? warp_sum(s) / (float)d : 0.f;
#pragma unroll 1
              for (int i = lane * 4; i < d; i += 128) {
                const float4 v = *reinterpret_cast<const float4*>(x + i);
                const float c0 = v.x - mean, c1 = v.y - mean, c2 = v.z - mean, c3 = v.w - mean;
                ss += (c0 * c0 + c1 * c1) + (c2 * c2 + c3 * c3);
              }
              const float rstd = 1.0f / sqrtf(warp_sum(ss) / (float)d + P.eps);
#pragma unroll 1
              for (int i = lane * 4; i < d; i += 128) {
                float4 v = *reinterpret_cast<const float4*>(x + i);
                const bool far = i >= 256;
                const float4 g4 = far ? __ldg(reinterpret_cast<const float4*>(g + i)) : i < 128 ? g0 : g1;
                const float4 b4 = far ? (b ? __ldg(reinterpret_cast<const float4*>(b + i)) : make_float4(0.f, 0.f, 0.f, 0.f)) : i < 128 ? b0 : b1;
                v.x = (v.x - mean) * rstd * g4.x + b4.x; v.y = (v.y - mean) * rstd * g4.y + b4.y;
                v.z = (v.z - mean) * rstd * g4.z + b4.z; v.w = (v.w - mean) * rstd * g4.w + b4.w;
                *reinterpret_cast<float4*>(sn + (size_t)warp * d + i) = v;
              }
            }
            __syncthreads();
          }
          unsigned long long best = 0ull;                              // LM head: of this lane's feature and row, over the warp's items
#pragma unroll 1
          for (int it = gw, slot = 0; it < items; it += NW) {
            const float *w0, *w1, *w2, *w3;                            // rows in the order of the features
            if (slots > 0) {
              if (tc::mbar_wait(reinterpret_cast<uint64_t*>(&S.landed[warp][slot]), (phases >> slot) & 1u, &S.abort, P.wait_limit)) {
                phases ^= 1u << slot;
                flying &= ~(1u << slot);
              }
              __syncwarp();
              w0 = ring + (size_t)slot * per; w1 = w0 + K; w2 = w1 + K; w3 = w2 + K;
              if (pairs) { const float* u = w1; w1 = w2; w2 = u; }
            } else {
              const float *p0, *p1;
              rows_of(L, kind, K, it, p0, p1);
              w0 = p0; w3 = p1 + K;
              if (pairs) { w1 = p1; w2 = p0 + K; }
              else { w1 = p0 + K; w2 = p1; }
              if (kind == ST_HEAD) {                                   // (a last item of fewer rows repeats its first)
                if (4 * it + 1 >= P.vocab) w1 = w0;
                if (4 * it + 2 >= P.vocab) w2 = w0;
                if (4 * it + 3 >= P.vocab) w3 = w0;
              }
            }
            float a[32];
#pragma unroll
            for (int i = 0; i < 32; ++i) a[i] = 0.f;
            auto fma_rows = [&](auto nt_) {   // (whole loads first: a branch per row would put every load's latency in the chain)
              constexpr int NT = decltype(nt_)::value;
#pragma unroll 2
              for (int k = lane * 4; k < K; k += 128) {
                const float4 q0 = *reinterpret_cast<const float4*>(w0 + k), q1 = *reinterpret_cast<const float4*>(w1 + k);
                const float4 q2 = *reinterpret_cast<const float4*>(w2 + k), q3 = *reinterpret_cast<const float4*>(w3 + k);
                float4 v[NT];
#pragma unroll
                for (int t = 0; t < NT; ++t) v[t] = *reinterpret_cast<const float4*>(act + (size_t)t * K + k);
#pragma unroll
                for (int t = 0; t < NT; ++t) {
                  a[t] = fmaf(q0.x, v[t].x, fmaf(q0.y, v[t].y, fmaf(q0.z, v[t].z, fmaf(q0.w, v[t].w, a[t]))));
                  a[8 + t] = fmaf(q1.x, v[t].x, fmaf(q1.y, v[t].y, fmaf(q1.z, v[t].z, fmaf(q1.w, v[t].w, a[8 + t]))));
                  a[16 + t] = fmaf(q2.x, v[t].x, fmaf(q2.y, v[t].y, fmaf(q2.z, v[t].z, fmaf(q2.w, v[t].w, a[16 + t]))));
                  a[24 + t] = fmaf(q3.x, v[t].x, fmaf(q3.y, v[t].y, fmaf(q3.z, v[t].z, fmaf(q3.w, v[t].w, a[24 + t]))));
                }
              }
            };
            if (rows <= 2) fma_rows(std::integral_constant<int, 2>());
            else if (rows <= 5) fma_rows(std::integral_constant<int, 5>());
            else fma_rows(std::integral_constant<int, 8>());
            float v = multi_sum<32>(a, lane);                          // feature fl, row tl
            if (slots > 0) {
              __syncwarp();
              if (it + slots * NW < items) fetch(L, kind, K, it + slots * NW, slot);
              slot = slot + 1 == slots ? 0 : slot + 1;
            }
            // ------------------------------------------------------ what becomes of it
            const int n = 4 * it + fl;
            if (kind == ST_HEAD) {
              if (on_row && n < P.vocab) {
                const unsigned long long k = argmax_key(v, (uint32_t)n);
                best = k > best ? k : best;
                if (P.logits) P.logits[(size_t)(off0 + r0 + tl) * P.vocab + n] = v;
              }
              continue;
            }
            if (kind == ST_UP && !glu) v = gelu_erf(v);
            // the item's four features of row tl, in all four of the row's lanes
            float4 v4;
            v4.x = __shfl_sync(0xffffffffu, v, tl); v4.y = __shfl_sync(0xffffffffu, v, 8 + tl);
            v4.z = __shfl_sync(0xffffffffu, v, 16 + tl); v4.w = __shfl_sync(0xffffffffu, v, 24 + tl);
            if (kind == ST_O || kind == ST_DOWN) {
              if (on_row) { const float4 x = *reinterpret_cast<const float4*>(sx + (size_t)tl * d + 4 * it); v4.x += x.x; v4.y += x.y; v4.z += x.z; v4.w += x.w; }
              __syncwarp();                                            // (all four lanes of a row read this CTA's copy before one of them writes it)
            }
            if (!on_row) continue;
            if (kind == ST_QKV) {
              const int at = qkv_at(it), m = at >> 28, col = at & 0x0fffffff;   // features col, col + half, col + 1, col + 1 + half
              if (P.rope && m < 2) {
                float cs[2], sn2[2];
#pragma unroll 1
                for (int e = 0; e < 2; ++e) {
                  const float inv = (float)exp2(-(double)(2 * (col % hd + e)) / (double)hd * log2((double)P.theta));
                  sincosf((float)S.pos[tl] * inv, &sn2[e], &cs[e]);
                }
                const float4 u = v4;
                v4.x = u.x * cs[0] - u.y * sn2[0]; v4.y = u.y * cs[0] + u.x * sn2[0];
                v4.z = u.z * cs[1] - u.w * sn2[1]; v4.w = u.w * cs[1] + u.z * sn2[1];
              }
              if (m == 0) {
                float* q = sq + (size_t)tl * nq + col;
                to_all2(q, v4.x * scale, v4.z * scale, NC, fl);
                to_all2(q + half, v4.y * scale, v4.w * scale, NC, fl);
              } else if (fl < 2) {
                float* c = (m == 1 ? L.kc : L.vc) + (size_t)S.kv[tl] * nkv + col + fl * half;
                __stcg(reinterpret_cast<float2*>(c), fl ? make_float2(v4.y, v4.w) : make_float2(v4.x, v4.z));
              }
            } else if (glu) {
              to_all2(sf + (size_t)tl * P.F + 2 * it, silu_f(v4.x) * v4.y, silu_f(v4.z) * v4.w, NC, fl);
            } else {
              float* dst = (kind == ST_UP ? sf + (size_t)tl * P.F : sx + (size_t)tl * d) + 4 * it;
              to_all4(dst, v4, NC, fl);
            }
          }
          if (kind == ST_HEAD && gw < items) {
#pragma unroll
            for (int o = 8; o < 32; o <<= 1) { const unsigned long long u = __shfl_xor_sync(0xffffffffu, best, o); best = u > best ? u : best; }
            if (on_row) to_all(&S.keys[tl][gw], best, NC, fl);
          }
        }
        if (st < 0 || gemm) {                                          // the ring is free: the next GEMM step's first items
          const int sn = st + 1 + (gemm && kind == ST_QKV), kn = sn == 5 * P.n_layers ? ST_HEAD : sn % 5;
          if (sn < n_steps) {
            const int Kn = depth_of(kn), n_slots = min(S_SLOTS, S_RING / 16 / Kn), n_items = items_of(kn);
            __syncwarp();
#pragma unroll 1
            for (int j = 0, it = gw; j < n_slots && it < n_items; ++j, it += NW) fetch(S.layers[min(sn / 5, P.n_layers - 1)], kn, Kn, it, j);
          }
        }
        __syncthreads();
        cl_arrive();
      }
      cl_wait();
      if (P.head_rows) {
        const int used = min(NW, (P.vocab + 3) / 4);                 // warps that had items
        if (warp < rows) {
          unsigned long long k = 0ull;
          for (int i = lane; i < used; i += 32) { const unsigned long long u = S.keys[warp][i]; k = u > k ? u : k; }
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) { const unsigned long long u = __shfl_xor_sync(0xffffffffu, k, o); k = u > k ? u : k; }
          if (lane == 0) S.result[r0 + warp] = argmax_key_index(k);
        }
      }
      __syncthreads();
    }
    if (P.mode == ROWS_DRAFT_FIRST && cta == 0 && tid == 0) P.draft_out[step] = S.result[T - 1];
  }
  if (*reinterpret_cast<volatile int*>(&S.abort)) {   // (never seen; bounds every wait all the same)
    if (tid == 0) *reinterpret_cast<volatile unsigned int*>(P.status + STATUS_ERROR) = 5u;   // STAIRS_ETIMEOUT
    for (int i = 0; i < S_SLOTS; ++i) {
      const long long t0 = clock64();
      while ((flying >> i & 1u) && !tc::mbar_try(reinterpret_cast<uint64_t*>(&S.landed[warp][i]), (phases >> i) & 1u) && (unsigned long long)(clock64() - t0) < P.wait_limit) {}
    }
  }
  // ---------------------------------------------------------------- accept
  if (P.mode == ROWS_VALIDATE && cta == 0) {
    for (int i = req0 + tid; i < req1; i += S_THREADS) {
      const int k = P.val_k[i], off = P.val_off[i] - off0, slot = P.val_req[i];
      int a = -1;
      for (int r = 0; r <= k; ++r) {
        const int tr = S.result[off + r];
        P.target_tokens[i * (P.k_max + 1) + r] = tr;
        if (a < 0 && r < k && P.draft[i * P.k_max + r] != tr) a = r;
      }
      if (a < 0) a = k;
      P.accept_len[i] = a;
      if (P.commit) {
        int* s = P.seq + (size_t)slot * P.max_seq_len;
        int w = P.n_seq[slot];
        for (int r = 0; r < a && w < P.max_seq_len; ++r) s[w++] = P.draft[i * P.k_max + r];
        if (w < P.max_seq_len) s[w++] = S.result[off + a];
        P.n_seq[slot] = w;
      }
    }
  }
}

}  // namespace small
}  // namespace stairs
