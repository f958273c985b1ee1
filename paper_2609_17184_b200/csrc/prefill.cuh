// Prompt passes of hundreds of positions (Algorithm 1, lines before the main loop): the prompt is the one place where the
// shared blocks see many token columns at once, so its GEMMs are bound by the tensor cores (three exact bf16 planes per
// fp32 activation) and not by the weight stream.  A pass carries up to PF_MAX_ROWS consecutive positions of one sequence at
// one recurrence; its rows need no row table (row i = position p0 + i, KV slot = position).
//
//   pf_prep_kernel     embedding rows (or states) -> fp32 stream, planes of x * gain, sum of squares
//   pf_concat_kernel   planes of [H; e] for the adapter of a Raven-style model
//   pf_gemm_kernel     QKV (+ 1/rms, RoPE, KV write), gate/up (+ 1/rms, SwiGLU, planes), O / down / adapter (k-split sums)
//   pf_reduce_kernel   k-split sums in split order + residual + planes of x * next gain + sum of squares
//   pf_attn_kernel     causal attention of the pass's rows over the cached keys and values
//
// A row's arithmetic is a function of its own operands and of the model's shapes: k-splits and the accumulation chains within them
// depend on the matrix alone, so results do not depend on how the prompt is cut into passes.
//
// Prompt of the 1.4B shape, wall clock of loopspec_prefill: 512 tokens 100 ms (passes of 32 rows; 61 ms with 64) -> 15.6 ms, 3001
// tokens 716 -> 110 ms; three-plane products at the measured GEMM peak would take 9 / 56 ms.
#pragma once
#include <cuda.h>

#include "attention.cuh"
#include "common.cuh"
#include "gemm.cuh"
#include "gemm_dec.cuh"
#include "linear_tc.cuh"

namespace ls {

constexpr int PF_MAX_ROWS = 1024;  // positions of one pass: at 1024 the persistent grid's last wave costs 5 to 14 % of a GEMM of
                                   // the 1.4B shape (21 to 35 % at 512), and a pass's activations still fit the L2
constexpr int PF_MAX_SPLIT = 4;
// k-splits of O, down and the adapter (few row blocks: 8 pairs at 2048 rows, on 74 pairs of CTAs): a function of K alone, at
// least eight 64-wide k-blocks each
__host__ __device__ inline int pf_splits(int K) {
  const int n = (K + 63) / 64 / 8;
  return n < 1 ? 1 : n > PF_MAX_SPLIT ? PF_MAX_SPLIT : n;
}

// ---- states -> planes ----------------------------------------------------------------------------------------------
struct PfPrepParams {
  const int* prompt;          // ids of the pass's positions (null: the rows' states are read from src)
  const __nv_bfloat16* embed; // [V][H]
  const float* src;           // [row][H]
  float* hid;                 // [row][H] written when the rows come from the embedding
  int H;
  const float* gain;          // null: no planes (the rows are only embedded)
  __nv_bfloat16* planes;      // [row][3][H]
  float* sumsq;               // [row]
};
// sum over the CTA (warp partials added in warp order), valid in thread 0
__device__ __forceinline__ float pf_block_sum(float v, float (&s_part)[8]) {
  v = warp_sum(v);
  if ((threadIdx.x & 31) == 0) s_part[threadIdx.x >> 5] = v;
  __syncthreads();
  float t = 0.f;
  if (threadIdx.x == 0)
    for (int w = 0; w < 8; ++w) t += s_part[w];
  return t;
}
__device__ __forceinline__ float pf_square_sum(float4 v) { return (v.x * v.x + v.y * v.y) + (v.z * v.z + v.w * v.w); }
__device__ __forceinline__ void pf_store_planes(__nv_bfloat16* row_planes, int H, int k, float4 v, const float* gain) {
  const float4 g = *reinterpret_cast<const float4*>(gain + k);
  store_split4(row_planes, H, k, make_float4(v.x * g.x, v.y * g.y, v.z * g.z, v.w * g.w));
}
// one CTA per row, four elements per thread and step (H is a multiple of 128)
__global__ void __launch_bounds__(256) pf_prep_kernel(const __grid_constant__ PfPrepParams p) {
  __shared__ float s_part[8];
  pdl_launch_dependents();
  pdl_wait();
  const int row = blockIdx.x;
  float ss = 0.f;
  for (int k = threadIdx.x * 4; k < p.H; k += 1024) {
    float4 v;
    if (p.prompt) {
      const uint2 w = *reinterpret_cast<const uint2*>(p.embed + (size_t)p.prompt[row] * p.H + k);
      v = make_float4(__uint_as_float(w.x << 16), __uint_as_float(w.x & 0xffff0000u), __uint_as_float(w.y << 16), __uint_as_float(w.y & 0xffff0000u));
      *reinterpret_cast<float4*>(p.hid + (size_t)row * p.H + k) = v;
    } else {
      v = *reinterpret_cast<const float4*>(p.src + (size_t)row * p.H + k);
    }
    if (!p.gain) continue;
    ss += pf_square_sum(v);
    pf_store_planes(p.planes + (size_t)row * 3 * p.H, p.H, k, v, p.gain);
  }
  if (!p.gain) return;
  ss = pf_block_sum(ss, s_part);
  if (threadIdx.x == 0) p.sumsq[row] = ss;
}

struct PfConcatParams {
  const float* hid;        // [row][H]
  float* e;                // [row][H] prelude outputs (written when first)
  int H, first;
  __nv_bfloat16* planes;   // [row][3][2 H]
};
__global__ void __launch_bounds__(256) pf_concat_kernel(const __grid_constant__ PfConcatParams p) {
  pdl_launch_dependents();
  pdl_wait();
  const int row = blockIdx.x;
  __nv_bfloat16* dst = p.planes + (size_t)row * 6 * p.H;
  for (int k = threadIdx.x * 4; k < p.H; k += 1024) {
    const float4 h = *reinterpret_cast<const float4*>(p.hid + (size_t)row * p.H + k);
    float4* ep = reinterpret_cast<float4*>(p.e + (size_t)row * p.H + k);
    const float4 ev = p.first ? h : *ep;
    if (p.first) *ep = h;
    store_split4(dst, 2 * p.H, k, h);
    store_split4(dst, 2 * p.H, p.H + k, ev);
  }
}

// ---- the GEMM ------------------------------------------------------------------------------------------------------
// y[token][n] = sum_k x[token][k] W[n][k] for a whole pass.  Bound by the tensor cores: 3 x 2 x rows x N x K operations, so
// everything here serves to keep tcgen05 fed.  A pair of CTAs (cluster of two, cta_group::2) owns 256 weight rows x 128 token
// columns: each CTA holds its 128 weight rows and half of the columns' operand, so a k-block of 64 costs an SM 40 KB of L2
// reads for 740 cycles of MMA (55 B per cycle; one CTA alone with 128 x 128 would need 83).  Per 16-wide k-step two MMAs:
// [hi | mid] as 256 columns (CTA 0 holds the hi rows, CTA 1 the mid rows of all 128 tokens) and lo as 128 columns that
// accumulate onto mid's - two chains, hi and (mid + lo), folded when the accumulator is read.  256 TMEM columns per
// accumulator, two accumulators in turn: the epilogue warps read one (chains of at most PG_SEG_MAX k-blocks, their sums kept in
// registers) while the MMAs of the next chain fill the other, and finish a tile under the first chains of the next (persistent
// CTAs, tiles dealt round robin, the token tiles of one weight block next to each other so that its weights come from HBM once).
// A k-block takes 740 cycles at 128 columns, 560 at 96 and 540 at 64, where the operands' way through the L2 bounds it (more
// stages change nothing); the MMAs are issued by a converged warp (see tc_elect_one: 840 cycles at any width before).  A pass of a
// few hundred tokens has one to three tiles per pair, so their width is chosen for even rounds (pg_tile_width), and what stands
// around the MMAs counts: 7000 cycles before the first (4000 of them after the predecessor's end) and 8000 to 10000 after the last.
// us per launch on the 1.4B shape: 368 tokens QKV 61 -> 27, gate/up 60 -> 44, down 31 -> 25; 512 tokens QKV 61 -> 36, gate/up 65 -> 60.
constexpr int PG_THREADS = 384;
constexpr int PG_TOK = 128;                        // token columns of a tile at most
constexpr int PG_WIDTHS = 3;                       // widths a tile can have: 128, 96 or 64 token columns (see pg_tile_width)
__host__ __device__ constexpr int pg_width(int i) { return PG_TOK - 32 * i; }
__host__ __device__ constexpr int pg_width_of(int cols) { return cols > 96 ? 0 : cols > 64 ? 1 : 2; }  // the narrowest that holds `cols`
constexpr int PG_A_BYTES = 128 * TC_BK * 2;        // a CTA's weight rows of a stage
constexpr int PG_B1_BYTES = PG_TOK * TC_BK * 2;    // hi (rank 0) or mid (rank 1) of all tokens
constexpr int PG_B2_BYTES = PG_TOK / 2 * TC_BK * 2;  // lo of half the tokens
constexpr int PG_STAGE_BYTES = PG_A_BYTES + PG_B1_BYTES + PG_B2_BYTES;
constexpr int PG_STAGES = 5;
constexpr int PG_ST_LD = 132;                      // floats per token of the epilogue's exchange buffer
constexpr int PG_ST_TOK = 16;                      // tokens exchanged at a time
constexpr int PG_SMEM = 1024 + PG_STAGES * PG_STAGE_BYTES + 2 * PG_ST_TOK * PG_ST_LD * 4;  // (an exchange buffer per epilogue team)
// k-blocks of one accumulation chain at most.  tcgen05 truncates its fp32 accumulator after every 16-wide step, so a sum's relative
// error grows with the length of its chain and not with K; the k-range of an item is cut into chains of its own, which the epilogue adds
// in order with rounded additions.  Relative error of the logits against float64 of one block of the 1.4B shape without its attention, 300
// tokens: whole k-ranges 2.6e-6, chains of 8 (QKV 6, O 4, down 5) 7.9e-7, of 4 6.1e-7; the passes of up to 64 rows, whose k-splits
// are such chains too, 9.1e-7.  Each chain costs the read of an accumulator: 70 tokens 6.97 -> 7.40 ms, 512
// 16.8 -> 16.8, 3001 111 -> 112.
constexpr int PG_SEG_MAX = 8;
enum { PG_QKV = 0, PG_SWIGLU = 1, PG_PART = 2 };

// The planes read by a GEMM as (k, token, plane), one pair of maps per tile width: boxes of the width (hi, mid) and of half of it (lo)
struct PgMaps {
  CUtensorMap x1[PG_WIDTHS], x2[PG_WIDTHS];
};
struct PfGemmParams {
  int n_rp, n_split;        // pairs of 128-row weight blocks, k-splits
  int tok, n_full, n_tail;  // token columns of a tile, tiles of that width, 1 when a narrower one is left over
  int n_kb, seg_kb;         // 64-wide k-blocks of the matrix, at most in one accumulation chain
  int n_tok, N;             // live rows of the pass, weight rows
  int* err;
  int err_code;
  const float* sumsq;       // [token]: columns are scaled by 1/sqrt(sumsq / H + eps)
  int H;
  float eps;
  float* part;              // PART: [split][token][N]
  long long split_stride;
  float* qbuf;              // QKV: [token][Hq]
  __nv_bfloat16* kv;        // QKV: this layer's and recurrence's plane [2][S][n_kv][slots][d]
  long long kv_sel_stride;
  int slots, n_kv_heads, n_q_heads, head_dim, seq, p0;
  const float2* rope;
  __nv_bfloat16* planes;    // SWIGLU: [token][3][F]
  int F;
};

__device__ __forceinline__ void pg_tma_2d(unsigned dst, const CUtensorMap* map, unsigned bar, int x, int y) {
  asm volatile("cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];" ::"r"(dst),
               "l"(reinterpret_cast<unsigned long long>(map)), "r"(bar), "r"(x), "r"(y)
               : "memory");
}
__device__ __forceinline__ void pg_tma_3d(unsigned dst, const CUtensorMap* map, unsigned bar, int x, int y, int z) {
  asm volatile("cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];" ::"r"(dst),
               "l"(reinterpret_cast<unsigned long long>(map)), "r"(bar), "r"(x), "r"(y), "r"(z)
               : "memory");
}
__device__ __forceinline__ void pg_mma(unsigned d_tmem, unsigned long long adesc, unsigned long long bdesc, unsigned idesc, unsigned accumulate) {
  asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\ttcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
               "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
               : "memory");
}
// arrives on the barrier at this offset in both CTAs of the pair once the MMAs issued so far are done
__device__ __forceinline__ void pg_commit(unsigned bar) {
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(bar), "h"((unsigned short)3)
               : "memory");
}
// Arrival that hands over nothing but an accumulator that has been read: no store of this thread needs to be visible with it (as a
// release at cluster scope it waited some 3500 cycles for the epilogue's stores)
__device__ __forceinline__ void pg_arrive_relaxed(unsigned addr) {
  asm volatile("mbarrier.arrive.relaxed.cluster.shared::cluster.b64 _, [%0];" ::"r"(addr) : "memory");
}
__device__ __forceinline__ void pg_cluster_sync() { asm volatile("barrier.cluster.arrive;\n\tbarrier.cluster.wait;" ::: "memory"); }
__device__ __forceinline__ void pg_team_sync(int team) { asm volatile("bar.sync %0, 128;" ::"r"(1 + team) : "memory"); }  // four warps of the epilogue
__device__ __forceinline__ void pg_ld16(unsigned (&w)[16], unsigned taddr) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
               : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]), "=r"(w[4]), "=r"(w[5]), "=r"(w[6]), "=r"(w[7]), "=r"(w[8]), "=r"(w[9]),
                 "=r"(w[10]), "=r"(w[11]), "=r"(w[12]), "=r"(w[13]), "=r"(w[14]), "=r"(w[15])
               : "r"(taddr)
               : "memory");
}

template <int EPI>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(PG_THREADS, 1)
    pf_gemm_kernel(const __grid_constant__ CUtensorMap map_w,   // weights: box 64 k x 128 rows; gate/up: (k, f, gate | up), box 64 x 64 x 2
                   const __grid_constant__ PgMaps maps,
                   const __grid_constant__ PfGemmParams p) {
  extern __shared__ unsigned char pg_smem_raw[];
  __shared__ __align__(8) unsigned long long s_full[PG_STAGES], s_empty[PG_STAGES], s_accf[2], s_acce[2];
  __shared__ unsigned s_tmem;
  __shared__ int s_fail;
  __shared__ float s_rstd[2][PG_TOK];

  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;  // (warp: uniform to the compiler)
  const unsigned rank = blockIdx.x & 1u;  // the pair's leader (rank 0) issues the MMAs and owns the full barriers
  const int cid = blockIdx.x >> 1, n_cl = gridDim.x >> 1;
  const unsigned base = (tc_smem_u32(pg_smem_raw) + 1023u) & ~1023u;
  const int n_full_items = p.n_rp * p.n_split * p.n_full, n_items = n_full_items + p.n_rp * p.n_split * p.n_tail;

  pdl_launch_dependents();
  if (tid == 0) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<unsigned long long>(&map_w)) : "memory");
    for (int s = 0; s < PG_STAGES; ++s) tc_mbar_init(tc_smem_u32(&s_full[s]), 1), tc_mbar_init(tc_smem_u32(&s_empty[s]), 1);
    for (int b = 0; b < 2; ++b) tc_mbar_init(tc_smem_u32(&s_accf[b]), 1), tc_mbar_init(tc_smem_u32(&s_acce[b]), 16);  // eight warps of each CTA
    s_fail = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  __syncthreads();
  // Both CTAs run and their barriers exist.  The allocation below is collective over the pair, so neither CTA may ask for it
  // before the other is known to be there (asked for at once, it was seen - rarely - never to return).
  pg_cluster_sync();
  if (warp == 2)
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tc_smem_u32(&s_tmem)), "r"(512u) : "memory");
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const unsigned tmem = s_tmem;

  // item -> (weight block pair, split, token tile): the full tiles first, token tiles fastest; the narrow ones of the leftover tokens
  // come last and fill what the full ones leave of the last round
  struct Item {
    int rp, sp, t0, live, kb_lo, n_kb, n_seg, cols;  // n_seg: accumulation chains of (nearly) equal length; cols: MMA columns of the tile
                                                     // (its live tokens rounded up to 32)
  };
  auto item_of = [&](int it) {
    Item r;
    int q, tt;
    if (it < n_full_items) q = it / p.n_full, tt = it - q * p.n_full;
    else q = it - n_full_items, tt = p.n_full;
    r.rp = q % p.n_rp, r.sp = q / p.n_rp;
    r.kb_lo = p.n_kb * r.sp / p.n_split;
    r.n_kb = p.n_kb * (r.sp + 1) / p.n_split - r.kb_lo;
    r.n_seg = (r.n_kb + p.seg_kb - 1) / p.seg_kb;
    r.t0 = tt * p.tok, r.live = min(p.tok, p.n_tok - r.t0);
    r.cols = (r.live + 31) & ~31;
    return r;
  };
  bool ok = true;
  auto wait = [&](unsigned long long* bar, unsigned parity) {  // bounded; after the first failure every later wait gives up at once
    if (!dg_wait(tc_smem_u32(bar), parity, ok ? TC_WAIT_CYCLES : 2000LL)) ok = false;
  };

  if (warp == 0) {
    if (lane == 0) {
      // ---- producer: this CTA's weight rows and its share of the planes; both CTAs complete on the leader's barrier --------
      auto load_w = [&](const Item& r, int kb, int s) {
        const unsigned bar = tc_smem_u32(&s_full[s]) & 0xFEFFFFFFu, a = base + s * PG_STAGE_BYTES;
        if (rank == 0) tc_mbar_expect_tx(tc_smem_u32(&s_full[s]), 2u * (PG_A_BYTES + pg_width(pg_width_of(r.cols)) * (3u * TC_BK)));
        if (EPI == PG_SWIGLU) pg_tma_3d(a, &map_w, bar, kb * TC_BK, (2 * r.rp + (int)rank) * 64, 0);
        else pg_tma_2d(a, &map_w, bar, kb * TC_BK, (2 * r.rp + (int)rank) * 128);
      };
      auto load_x = [&](const Item& r, int kb, int s) {
        const unsigned bar = tc_smem_u32(&s_full[s]) & 0xFEFFFFFFu, b = base + s * PG_STAGE_BYTES + PG_A_BYTES;
        const int w = pg_width_of(r.cols);
        pg_tma_3d(b, &maps.x1[w], bar, kb * TC_BK, r.t0, (int)rank);
        pg_tma_3d(b + PG_B1_BYTES, &maps.x2[w], bar, kb * TC_BK, r.t0 + (int)rank * (r.cols >> 1), 2);
      };
      // the first ring-full of weights is requested ahead of the predecessor's completion
      int pre = 0;
      if (cid < n_items) {
        const Item r = item_of(cid);
        for (; pre < min(PG_STAGES, r.n_kb); ++pre) load_w(r, r.kb_lo + pre, pre);
      }
      pdl_wait();
      int s = 0, u = 0;
      unsigned par = 1;  // (the first use of a stage finds it free)
      for (int it = cid; it < n_items; it += n_cl) {
        const Item r = item_of(it);
        for (int kb = 0; kb < r.n_kb; ++kb, ++u) {
          if (u >= PG_STAGES) wait(&s_empty[s], par);
          if (u >= pre) load_w(r, r.kb_lo + kb, s);
          load_x(r, r.kb_lo + kb, s);
          if (++s == PG_STAGES) s = 0, par ^= 1u;
        }
      }
      for (int i = 0; i < min(u, PG_STAGES); ++i) {  // the leader's last arrivals on this CTA's barriers have landed before it may exit
        if (u < PG_STAGES) wait(&s_empty[i], 0);
        else {
          wait(&s_empty[s], par);
          if (++s == PG_STAGES) s = 0, par ^= 1u;
        }
      }
      if (!ok) s_fail = 1, *p.err = p.err_code;
    }
  } else if (warp == 1) {
    if (rank == 0) {
      // ---- MMA issuer of the pair: the warp walks the k-blocks together, one elected lane issues (see tc_elect_one) ------------
      const unsigned long long desc0 = tc_smem_desc(0);
      int s = 0, n = 0;  // n: segments so far
      unsigned par = 0;
      for (int it = cid; it < n_items; it += n_cl) {
        const Item r = item_of(it);
        const unsigned idesc1 = tc_idesc(256, 2 * r.cols), idesc2 = tc_idesc(256, r.cols);
        for (int sg = 0, kb = 0; sg < r.n_seg; ++sg, ++n) {
          const int buf = n & 1, uses = n >> 1, first = kb, end = r.n_kb * (sg + 1) / r.n_seg;
          if (uses > 0) wait(&s_acce[buf], (uses - 1) & 1);
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const unsigned d = tmem + buf * 256;
          for (; kb < end; ++kb) {
            wait(&s_full[s], par);
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            if (tc_elect_one()) {
              const unsigned a = base + s * PG_STAGE_BYTES, b1 = a + PG_A_BYTES, b2 = b1 + PG_B1_BYTES;
              const unsigned long long ad = desc0 | ((a >> 4) & 0x3FFF), bd1 = desc0 | ((b1 >> 4) & 0x3FFF), bd2 = desc0 | ((b2 >> 4) & 0x3FFF);
#pragma unroll
              for (int ks = 0; ks < TC_BK / 16; ++ks) {
                pg_mma(d, ad + 2 * ks, bd1 + 2 * ks, idesc1, kb > first || ks > 0);
                pg_mma(d + r.cols, ad + 2 * ks, bd2 + 2 * ks, idesc2, 1);
              }
              pg_commit(tc_smem_u32(&s_empty[s]));
              if (kb == end - 1) pg_commit(tc_smem_u32(&s_accf[buf]));
            }
            __syncwarp();
            if (++s == PG_STAGES) s = 0, par ^= 1u;
          }
        }
      }
      if (!ok && lane == 0) s_fail = 1, *p.err = p.err_code;
    }
  } else if (warp >= 4) {
    // ---- epilogue: thread = weight row of this CTA's block.  Two teams of four warps take 16 tokens each in turn: with one, the
    // epilogue of a QKV tile (its rotary factors waited for one by one) took as long as two tiles of MMAs, and a pass of a few
    // hundred tokens has one or two tiles per pair to hide it behind [QKV of 400 tokens: 61 us with both] ----------------
    pdl_wait();
    const int team = (warp - 4) >> 2, ew = warp & 3, j = (tid - 128) & 127;
    const unsigned lane_off = (unsigned)(ew * 32) << 16;
    float* const sx = reinterpret_cast<float*>(pg_smem_raw + (base - tc_smem_u32(pg_smem_raw)) + PG_STAGES * PG_STAGE_BYTES) + team * (PG_ST_TOK * PG_ST_LD);
    int n = 0;  // segments so far
    for (int it = cid; it < n_items; it += n_cl) {
      const Item r = item_of(it);
      const int t0 = r.t0, live = r.live;
      const int n0 = (2 * r.rp + (int)rank) * (EPI == PG_SWIGLU ? 64 : 128);
      // QKV: a thread's rotary pair, its eight tokens of a step, and their rotary factors (requested a step ahead)
      const int d = p.head_dim, hd2 = d >> 1, Hq = p.n_q_heads * d, Hk = p.n_kv_heads * d;
      const int region = n0 < Hq ? 0 : (n0 < Hq + Hk ? 1 : 2);
      const int rbase = region == 0 ? 0 : (region == 1 ? Hq : Hq + Hk);
      const int pj = j & 63, hh = EPI == PG_QKV ? pj / hd2 : 0, i = pj - hh * hd2, head = EPI == PG_QKV ? (n0 - rbase) / d + hh : 0, tq = (j >> 6) * 8;
      float2 cs[8];
      auto load_cs = [&](int c0) {
#pragma unroll
        for (int q = 0; q < 8; ++q)
          cs[q] = region < 2 && c0 + tq + q < live ? p.rope[(size_t)(p.p0 + t0 + c0 + tq + q) * hd2 + i] : make_float2(1.f, 0.f);
      };
      if (EPI == PG_QKV) load_cs(team * PG_ST_TOK);
      if (EPI != PG_PART) {
        pg_team_sync(team);  // the previous tile's readers of s_rstd are done
        if (j < live) s_rstd[team][j] = 1.0f / sqrtf(p.sumsq[t0 + j] / (float)p.H + p.eps);
      }
      // the segments' sums, added in order: this thread's weight row, its team's token columns
      constexpr int STEPS = PG_TOK / 2 / PG_ST_TOK;
      float acc[STEPS][PG_ST_TOK];
      for (int sg = 0; sg < r.n_seg; ++sg, ++n) {
        const int buf = n & 1, uses = n >> 1;
        wait(&s_accf[buf], uses & 1);
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
        for (int q = 0; q < STEPS; ++q) {
          const int c0 = (2 * q + team) * PG_ST_TOK;
          if (c0 < live) {
            unsigned hi[16], ml[16];
            pg_ld16(hi, tmem + lane_off + buf * 256 + c0);
            pg_ld16(ml, tmem + lane_off + buf * 256 + r.cols + c0);
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
            for (int c = 0; c < PG_ST_TOK; ++c) {
              const float v = __uint_as_float(hi[c]) + __uint_as_float(ml[c]);
              acc[q][c] = sg == 0 ? v : acc[q][c] + v;
            }
          }
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncwarp();
        if (lane == 0) pg_arrive_relaxed(dg_mapa(tc_smem_u32(&s_acce[buf]), 0));  // the accumulator may be overwritten
      }
      if constexpr (EPI == PG_PART) {
        if (n0 + j < p.N) {
#pragma unroll
          for (int q = 0; q < STEPS; ++q) {
            const int c0 = (2 * q + team) * PG_ST_TOK;
            float* out = p.part + (size_t)r.sp * p.split_stride + (size_t)(t0 + c0) * p.N + n0 + j;
#pragma unroll
            for (int c = 0; c < PG_ST_TOK; ++c)
              if (c0 + c < live) out[(size_t)c * p.N] = acc[q][c];
          }
        }
      } else {
        for (int c0 = team * PG_ST_TOK; c0 < live; c0 += 2 * PG_ST_TOK) {
          pg_team_sync(team);  // the readers of the step before are done
#pragma unroll
          for (int q = 0; q < STEPS; ++q)  // (registers are addressed by constants)
            if (c0 == (2 * q + team) * PG_ST_TOK) {
#pragma unroll
              for (int c = 0; c < PG_ST_TOK; ++c) sx[c * PG_ST_LD + j] = acc[q][c];
            }
          pg_team_sync(team);
          if (EPI == PG_SWIGLU) {  // two neighbouring features, four tokens per thread
            const int f2 = 2 * lane, f = n0 + f2;
            if (f < p.F) {
#pragma unroll
              for (int q = 0; q < 4; ++q) {
                const int c = ew * 4 + q;
                const float rs = s_rstd[team][c0 + c];
                const float2 gt = *reinterpret_cast<const float2*>(sx + c * PG_ST_LD + f2), up = *reinterpret_cast<const float2*>(sx + c * PG_ST_LD + 64 + f2);
                const float g0 = gt.x * rs, g1 = gt.y * rs;
                const float y0 = g0 / (1.0f + expf(-g0)) * (up.x * rs), y1 = g1 / (1.0f + expf(-g1)) * (up.y * rs);
                if (c0 + c < live) store_split2(p.planes + (size_t)(t0 + c0 + c) * 3 * p.F, p.F, f, y0, y1);
              }
            }
          } else if (n0 < p.N) {  // QKV: a rotary pair, eight tokens per thread
            float2 y[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) {
              const float rs = s_rstd[team][c0 + tq + q];
              const float x1 = sx[(tq + q) * PG_ST_LD + hh * d + i] * rs, x2 = sx[(tq + q) * PG_ST_LD + hh * d + i + hd2] * rs;
              y[q] = region < 2 ? make_float2(x1 * cs[q].x - x2 * cs[q].y, x2 * cs[q].x + x1 * cs[q].y) : make_float2(x1, x2);
            }
            load_cs(c0 + 2 * PG_ST_TOK);
#pragma unroll
            for (int q = 0; q < 8; ++q) {
              const int c = c0 + tq + q;
              if (c >= live) continue;
              if (region == 0) {
                float* qd = p.qbuf + (size_t)(t0 + c) * Hq + head * d + i;
                qd[0] = y[q].x, qd[hd2] = y[q].y;
              } else {
                __nv_bfloat16* dst = p.kv + (size_t)(region - 1) * p.kv_sel_stride + ((size_t)(p.seq * p.n_kv_heads + head) * p.slots + p.p0 + t0 + c) * d + i;
                dst[0] = __float2bfloat16_rn(y[q].x), dst[hd2] = __float2bfloat16_rn(y[q].y);
              }
            }
          }
        }
      }
    }
    if (!ok && lane == 0) s_fail = 1, *p.err = p.err_code;
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (tid == 0 && s_fail) {  // a wait gave up: copies may still be in flight; give them a bounded time before the memory goes
    const long long t0 = clock64();
    while (clock64() - t0 < 2000000LL) {
    }
  }
  __syncthreads();
  pg_cluster_sync();  // the partner still reads this CTA's memory until here
  if (warp == 2) {
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
  }
}

// ---- k-split sums + residual + planes of the next consumer's input ------------------------------------------------------
struct PfReduceParams {
  const float* part;       // [split][token][H]
  int n_split;
  long long split_stride;
  const float* hid_in;     // null: the sums replace the stream (the adapter of a Raven-style model)
  float* hid_out;          // [token][H]
  int H;
  const float* gain;       // of the norm that reads the stream next (null: nobody reads planes)
  __nv_bfloat16* planes;
  float* sumsq;            // [token]
};
// Bound by its bytes (per row: n_split + 2 fp32 rows and three bf16 planes, mostly in the L2): one CTA per row, 16-byte
// accesses, every load of a step in flight at once.
__global__ void __launch_bounds__(256) pf_reduce_kernel(const __grid_constant__ PfReduceParams p) {
  __shared__ float s_part[8];
  pdl_launch_dependents();
  pdl_wait();
  const int row = blockIdx.x;
  float ss = 0.f;
  for (int k = threadIdx.x * 4; k < p.H; k += 1024) {
    const size_t at = (size_t)row * p.H + k;
    float4 t[PF_MAX_SPLIT];
#pragma unroll
    for (int s = 0; s < PF_MAX_SPLIT; ++s)
      if (s < p.n_split) t[s] = __ldcg(reinterpret_cast<const float4*>(p.part + (size_t)s * p.split_stride + at));
    float4 v = p.hid_in ? *reinterpret_cast<const float4*>(p.hid_in + at) : make_float4(0.f, 0.f, 0.f, 0.f);
    float4 y = t[0];
#pragma unroll
    for (int s = 1; s < PF_MAX_SPLIT; ++s)
      if (s < p.n_split) y.x += t[s].x, y.y += t[s].y, y.z += t[s].z, y.w += t[s].w;
    v.x += y.x, v.y += y.y, v.z += y.z, v.w += y.w;
    *reinterpret_cast<float4*>(p.hid_out + at) = v;
    if (!p.gain) continue;
    ss += pf_square_sum(v);
    pf_store_planes(p.planes + (size_t)row * 3 * p.H, p.H, k, v, p.gain);
  }
  if (!p.gain) return;
  ss = pf_block_sum(ss, s_part);
  if (threadIdx.x == 0) p.sumsq[row] = ss;
}

// ---- attention ---------------------------------------------------------------------------------------------------------
// A CTA owns 64 rows of the pass and one query head.  Two groups of four warps (16 rows per warp) walk the keys 64 at a time, one the
// even chunks and one the odd; every row keeps a running softmax per group, and the two are folded at the end.  Both
// contractions are mma.sync on exact three-plane splits, chains hi and (mid + lo) of one chunk folded in fp32 (a row's result
// depends on its own prefix only: chunks lie at absolute positions).  The softmax weights never leave registers: an accumulator
// fragment of the scores is the A fragment of the second contraction.  Keys and values are double-buffered (cp.async) per
// group; rows of shared memory are swizzled in 16-byte pieces so that ldmatrix is free of bank conflicts.  Blocks with the
// longest prefixes start first.  A chunk is a chain of some 7800 cycles of one warp against 3100 of its MMAs, so a prompt of a few
// hundred positions is bound by the longest block's chain, which the two groups halve.
// Of the 1.4B shape, one group of four warps -> two: 512 positions 36 -> 28 us, the last pass of 3001 positions 237 -> 207 us.
constexpr int PFA_ROWS = 64, PFA_KEYS = 64, PFA_GROUPS = 2, PFA_THREADS = PFA_GROUPS * 128;
template <int D>
struct PfaCfg {
  static constexpr int ROWB = D * 2;                                // bytes of a row of Q, K, V
  static constexpr int Q_BYTES = 3 * PFA_ROWS * ROWB, KV_BYTES = PFA_KEYS * ROWB;
  static constexpr int SMEM_BYTES = Q_BYTES + PFA_GROUPS * 4 * KV_BYTES;  // Q planes, two buffers of K and V per group
  static constexpr int FOLD_LD = D + 4;                             // floats per row of the fold's buffer (over a group's K and V)
  static_assert(PFA_ROWS * FOLD_LD * 4 <= 4 * KV_BYTES, "the second group's rows fit its buffers");
};
struct PfAttnParams {
  const float* qbuf;         // [row][n_q_heads * D], rotary applied, unscaled
  __nv_bfloat16* aplanes;    // [row][3][n_q_heads * D]
  const __nv_bfloat16* k;    // the sequence's keys of this layer and recurrence [n_kv][slots][D]
  const __nv_bfloat16* v;
  int n_rows, p0, slots, n_kv_heads, n_q_heads;
  float scale;
};

template <int D>
__global__ void __launch_bounds__(PFA_THREADS, 1) pf_attn_kernel(const __grid_constant__ PfAttnParams p) {
  using C = PfaCfg<D>;
  constexpr int PCS = D / 8;  // 16-byte pieces per row
  extern __shared__ __align__(128) unsigned char pfa_smem[];
  const int tid = threadIdx.x, grp = tid >> 7, gtid = tid & 127, warp = (tid >> 5) & 3, lane = tid & 31, g = lane >> 2, t = lane & 3;
  const unsigned sq = (unsigned)__cvta_generic_to_shared(pfa_smem), sk = sq + C::Q_BYTES + grp * 4 * C::KV_BYTES, sv = sk + 2 * C::KV_BYTES;
  auto group_sync = [&]() { asm volatile("bar.sync %0, 128;" ::"r"(1 + grp) : "memory"); };
  pdl_launch_dependents();
  const int h = blockIdx.x % p.n_q_heads, n_blocks = (p.n_rows + PFA_ROWS - 1) / PFA_ROWS;
  const int blk = n_blocks - 1 - blockIdx.x / p.n_q_heads;
  const int row0 = blk * PFA_ROWS, rows_here = min(PFA_ROWS, p.n_rows - row0);
  const int HQ = p.n_q_heads * D, kvh = h / (p.n_q_heads / p.n_kv_heads);
  const int n_keys = p.p0 + row0 + rows_here;            // keys the block's last row sees
  const int n_chunks = (n_keys + PFA_KEYS - 1) / PFA_KEYS;
  const __nv_bfloat16* Kb = p.k + (size_t)kvh * p.slots * D;
  const __nv_bfloat16* Vb = p.v + (size_t)kvh * p.slots * D;
  auto piece = [](int row, int c) { return (unsigned)(row * C::ROWB + ((c ^ (row & 7)) << 4)); };
  auto load_chunk = [&](int chunk, int b) {
    const int k0 = chunk * PFA_KEYS;
#pragma unroll
    for (int i = 0; i < PFA_KEYS * PCS / 128; ++i) {
      const int idx = gtid + i * 128, key = idx / PCS, c = idx % PCS;
      const bool live = k0 + key < n_keys;
      const size_t off = (size_t)(live ? k0 + key : 0) * D + c * 8;
      const int n = live ? 16 : 0;  // keys beyond the block's last position: zeros
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(sk + b * C::KV_BYTES + piece(key, c)), "l"(Kb + off), "r"(n) : "memory");
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(sv + b * C::KV_BYTES + piece(key, c)), "l"(Vb + off), "r"(n) : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  pdl_wait();
  if (grp < n_chunks) load_chunk(grp, 0);
  // the block's queries, split into three planes (rows the pass does not have: zeros)
  for (int idx = tid; idx < PFA_ROWS * PCS; idx += PFA_THREADS) {
    const int lr = idx / PCS, c = idx % PCS;
    float x[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    if (lr < rows_here) {
      const float4* src = reinterpret_cast<const float4*>(p.qbuf + (size_t)(row0 + lr) * HQ + (size_t)h * D + c * 8);
      const float4 a = src[0], b = src[1];
      x[0] = a.x, x[1] = a.y, x[2] = a.z, x[3] = a.w, x[4] = b.x, x[5] = b.y, x[6] = b.z, x[7] = b.w;
    }
    unsigned s[4][3];
#pragma unroll
    for (int i = 0; i < 4; ++i) split3_pair(x[2 * i], x[2 * i + 1], s[i]);
#pragma unroll
    for (int pl = 0; pl < 3; ++pl)
      *reinterpret_cast<uint4*>(pfa_smem + pl * PFA_ROWS * C::ROWB + piece(lr, c)) = make_uint4(s[0][pl], s[1][pl], s[2][pl], s[3][pl]);
  }
  __syncthreads();
  float o[D / 8][4], m[2] = {-INFINITY, -INFINITY}, l[2] = {0.f, 0.f};
#pragma unroll
  for (int j = 0; j < D / 8; ++j)
#pragma unroll
    for (int i = 0; i < 4; ++i) o[j][i] = 0.f;
  const int wr = warp * 16;                 // this warp's first row of the block
  const int last_pos = p.p0 + row0 + wr + 15;  // ... and the last position any of them has
  // ldmatrix lane addresses: A tiles (16 x 16): rows lane & 15, piece half lane >> 4; B tiles of K (two 8-key tiles x 16 dims):
  // keys (lane & 7) + 8 (lane >> 4), piece half (lane >> 3) & 1; V, transposed: keys lane & 15, piece half lane >> 4
  for (int chunk = grp; chunk < n_chunks; chunk += PFA_GROUPS) {
    const int b = (chunk / PFA_GROUPS) & 1, k0 = chunk * PFA_KEYS;
    if (chunk + PFA_GROUPS < n_chunks) {
      load_chunk(chunk + PFA_GROUPS, b ^ 1);
      asm volatile("cp.async.wait_group 1;" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    group_sync();
    if (k0 <= last_pos) {  // (uniform over the warp) some row of the warp sees this chunk
      float s0[8][4], s1[8][4];
#pragma unroll
      for (int j = 0; j < 8; ++j)
#pragma unroll
        for (int i = 0; i < 4; ++i) s0[j][i] = s1[j][i] = 0.f;
#pragma unroll 2
      for (int ks = 0; ks < D / 16; ++ks) {
        unsigned a[3][4];
#pragma unroll
        for (int pl = 0; pl < 3; ++pl) att_ldsm4(a[pl], sq + pl * PFA_ROWS * C::ROWB + piece(wr + (lane & 15), 2 * ks + (lane >> 4)));
#pragma unroll
        for (int jj = 0; jj < 4; ++jj) {  // two tiles of eight keys
          unsigned kb[4];
          att_ldsm4(kb, sk + b * C::KV_BYTES + piece(16 * jj + (lane & 7) + 8 * (lane >> 4), 2 * ks + ((lane >> 3) & 1)));
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            att_mma(s0[2 * jj + e], a[0], kb[2 * e], kb[2 * e + 1]);
            att_mma(s1[2 * jj + e], a[1], kb[2 * e], kb[2 * e + 1]);
            att_mma(s1[2 * jj + e], a[2], kb[2 * e], kb[2 * e + 1]);
          }
        }
      }
      // scores, causal mask, running maximum of rows g and g + 8
      const bool edge = k0 + PFA_KEYS - 1 > p.p0 + row0 + wr;  // some key of the chunk lies beyond some row of the warp
      float mn[2] = {m[0], m[1]};
#pragma unroll
      for (int j = 0; j < 8; ++j)
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int hf = i >> 1;
          float sv_ = (s0[j][i] + s1[j][i]) * p.scale;
          if (edge && k0 + 8 * j + 2 * t + (i & 1) > p.p0 + row0 + wr + g + 8 * hf) sv_ = -INFINITY;
          s0[j][i] = sv_;
          mn[hf] = fmaxf(mn[hf], sv_);
        }
      float wa[2], m0[2], lc[2] = {0.f, 0.f};
#pragma unroll
      for (int hf = 0; hf < 2; ++hf) {
        mn[hf] = fmaxf(mn[hf], __shfl_xor_sync(0xffffffffu, mn[hf], 1));
        mn[hf] = fmaxf(mn[hf], __shfl_xor_sync(0xffffffffu, mn[hf], 2));
        wa[hf] = m[hf] == -INFINITY ? 0.f : expf(m[hf] - mn[hf]);
        m[hf] = mn[hf];
        m0[hf] = mn[hf] == -INFINITY ? 0.f : mn[hf];  // (a row that sees none of the group's chunks so far: every weight is zero)
      }
      // weights, split into three planes as A fragments: keys 16 kk + 2 t (+ 1) from tile 2 kk, + 8 from tile 2 kk + 1
      unsigned pa[PFA_KEYS / 16][3][4];
#pragma unroll
      for (int j = 0; j < 8; ++j)
#pragma unroll
        for (int hf = 0; hf < 2; ++hf) {
          const float e0 = expf(s0[j][2 * hf] - m0[hf]), e1 = expf(s0[j][2 * hf + 1] - m0[hf]);
          lc[hf] += e0 + e1;
          unsigned w[3];
          split3_pair(e0, e1, w);
#pragma unroll
          for (int pl = 0; pl < 3; ++pl) pa[j >> 1][pl][hf + 2 * (j & 1)] = w[pl];
        }
#pragma unroll
      for (int hf = 0; hf < 2; ++hf) {
        lc[hf] += __shfl_xor_sync(0xffffffffu, lc[hf], 1);
        lc[hf] += __shfl_xor_sync(0xffffffffu, lc[hf], 2);
        l[hf] = fmaf(l[hf], wa[hf], lc[hf]);
      }
      // weighted values: 16 dims at a time (two tiles of eight)
#pragma unroll
      for (int dt = 0; dt < D / 16; ++dt) {
        float a0[2][4], a1[2][4];
#pragma unroll
        for (int e = 0; e < 2; ++e)
#pragma unroll
          for (int i = 0; i < 4; ++i) a0[e][i] = a1[e][i] = 0.f;
#pragma unroll
        for (int kk = 0; kk < PFA_KEYS / 16; ++kk) {
          unsigned vb[4];
          att_ldsm4_t(vb, sv + b * C::KV_BYTES + piece(16 * kk + (lane & 15), 2 * dt + (lane >> 4)));
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            att_mma(a0[e], pa[kk][0], vb[2 * e], vb[2 * e + 1]);
            att_mma(a1[e], pa[kk][1], vb[2 * e], vb[2 * e + 1]);
            att_mma(a1[e], pa[kk][2], vb[2 * e], vb[2 * e + 1]);
          }
        }
#pragma unroll
        for (int e = 0; e < 2; ++e)
#pragma unroll
          for (int i = 0; i < 4; ++i) o[2 * dt + e][i] = fmaf(o[2 * dt + e][i], wa[i >> 1], a0[e][i] + a1[e][i]);
      }
    }
    group_sync();  // the buffer may be refilled
  }
  // ---- the odd chunks' sums join the even chunks' ----
  float* const fold = reinterpret_cast<float*>(pfa_smem + C::Q_BYTES + 4 * C::KV_BYTES);
  if (grp == 1) {  // (all of this group's reads of its buffers are behind its last barrier)
#pragma unroll
    for (int hf = 0; hf < 2; ++hf) {
      float* row = fold + (wr + g + 8 * hf) * C::FOLD_LD;
      if (t == 0) row[D] = m[hf], row[D + 1] = l[hf];
#pragma unroll
      for (int j = 0; j < D / 8; ++j) *reinterpret_cast<float2*>(row + 8 * j + 2 * t) = make_float2(o[j][2 * hf], o[j][2 * hf + 1]);
    }
  }
  __syncthreads();
  if (grp == 1) return;
#pragma unroll
  for (int hf = 0; hf < 2; ++hf) {
    const int lr = wr + g + 8 * hf;
    if (lr >= rows_here) continue;
    const float* row = fold + lr * C::FOLD_LD;
    const float m1 = row[D], mx = fmaxf(m[hf], m1);  // (key 0 is among the even chunks' and visible to every row: finite)
    const float w0 = expf(m[hf] - mx), w1 = m1 == -INFINITY ? 0.f : expf(m1 - mx), mass = fmaf(l[hf], w0, row[D + 1] * w1);
    __nv_bfloat16* dst = p.aplanes + (size_t)(row0 + lr) * 3 * HQ;
#pragma unroll
    for (int j = 0; j < D / 8; ++j) {
      const float2 o1 = *reinterpret_cast<const float2*>(row + 8 * j + 2 * t);
      store_split2(dst, HQ, h * D + 8 * j + 2 * t, fmaf(o[j][2 * hf], w0, o1.x * w1) / mass, fmaf(o[j][2 * hf + 1], w0, o1.y * w1) / mass);
    }
  }
}

// ---- the prompt's last row, ready for the readout: one table row, its planes of x * final gain, its sum of squares ----------
struct PfReadoutParams {
  RowTable* tab;
  const float* row;        // [H] the last position's state after R recurrences (and the post-layers' blocks)
  int H, seq, pos, R, hid_idx, logit_idx;
  const float* gain;
  __nv_bfloat16* planes;   // [3][H]: column 0 of the decode passes' planes
  float* sumsq;
};
__global__ void __launch_bounds__(256) pf_readout_kernel(const __grid_constant__ PfReadoutParams p) {
  __shared__ float s_part[8];
  pdl_wait();
  float ss = 0.f;
  for (int k = threadIdx.x * 4; k < p.H; k += 1024) {
    const float4 v = *reinterpret_cast<const float4*>(p.row + k);
    ss += pf_square_sum(v);
    pf_store_planes(p.planes, p.H, k, v, p.gain);
  }
  ss = pf_block_sum(ss, s_part);
  if (threadIdx.x != 0) return;
  p.sumsq[0] = ss;
  RowTable& t = *p.tab;
  t.n_rows = 1, t.n_readout = 1, t.attn_items = 0, t.chunk_start[0] = t.chunk_start[1] = 0;
  t.seq[0] = p.seq, t.r[0] = p.R, t.pos[0] = p.pos, t.kv_slot[0] = p.pos, t.n_canon[0] = p.pos + 1, t.n_spec[0] = 0, t.n_safe[0] = p.pos;
  t.hid_idx[0] = p.hid_idx, t.node[0] = -1, t.src_hid[0] = -1, t.readout[0] = RO_TARGET, t.logit_idx[0] = p.logit_idx, t.ro_rows[0] = 0;
}

}  // namespace ls
