// Decode attention over the depth-indexed KV cache (App. B "KV Cache Management"): a row advanced to
// recurrence r attends to the keys/values that its prefix produced at the SAME recurrence r -- the
// committed slots [0, n_canon) of plane r plus the speculative slots of its uncommitted ancestors and itself.
//
// Three kernels, by regime:
//   attn_kernel          work item = (row, kv head, chunk of ATT_CHUNK key positions): one CTA each, every chunk in parallel, for
//                        the few rows and short prefixes of a single sequence's decode pass (latency matters);
//   attn_warp_kernel     work item = (row, kv head, run of chunks): one warp each, on the tensor cores; long prefixes and
//                        contexts of several sequences (bandwidth and the number of items matter; the line: att_line).
//                        Logits of both against float64 agree in three digits (2410 positions of the 256-wide model: 3.65e-5);
//   attn_prefill_mma_kernel  work item = (query head, block of rows, run of chunks) for the consecutive positions of a prefill
//                        pass, which share their keys and values.
// Chunks and runs are cut at fixed absolute positions (or as a function of the row's own context) and folded in
// ascending order, so a row's result does not depend on what else is in the pass.
#pragma once
#include "common.cuh"

namespace ls {

// 16-byte asynchronous copy into shared memory; !valid: the 16 bytes are zero-filled and nothing is read
__device__ __forceinline__ void cp_async16_zfill(void* smem_dst, const void* gsrc, bool valid) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(smem_dst);
  const int n = valid ? 16 : 0;
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(gsrc), "r"(n) : "memory");
}

constexpr int ATT_THREADS = 256;  // 8 warps per work item; at most 64 registers per thread so that the
                                   // neighbouring GEMM kernels' CTAs can be resident (and prefetching) alongside

struct AttnParams {
  const RowTable* tab;
  const float* qbuf;          // [row][n_q_heads * d], rotary applied, unscaled
  __nv_bfloat16* aplanes;     // out: three bf16 planes per row [row][3][n_q_heads * d]
  const __nv_bfloat16* kv;    // this layer's pool [R][2][S][n_kv][slots][d]
  long long kv_plane_stride, kv_sel_stride;
  int slots, n_kv_heads, n_q_heads;
  float scale;                // 1/sqrt(d)
  float* part;                // [row][n_kv][max_chunks][G][D + 2]
  int max_chunks;
  int* counters;              // [row][n_kv]
  long long* dbg;             // tuning aid: cycle stamps of CTA 0 / thread 0 (null in production)
  unsigned long long* tl;     // tuning aid: kernel timeline (null in production)
  int tl_id;
};

template <int D, int G>
__global__ void __launch_bounds__(ATT_THREADS, 4) attn_kernel(const __grid_constant__ AttnParams p) {
  constexpr int LPP = D / 8;            // lanes per key position (8 bf16 = 16 bytes per lane)
  constexpr int PPW = 32 / LPP;         // positions per warp per load
  constexpr int PPR = PPW * (ATT_THREADS / 32);  // positions per round of the whole CTA
  constexpr int NPOS = ATT_CHUNK + MAX_SPEC;     // the last chunk of a row also carries its speculative slots
  constexpr int ROUNDS = (NPOS + PPR - 1) / PPR;
  constexpr int PSTRIDE = D + 2;

  __shared__ float s_score[G][ROUNDS * PPR];
  __shared__ float s_red[ATT_THREADS / 32][G][D];
  __shared__ float s_stat[G][2];
  __shared__ int s_last;

  int dbg_n = 0;
  auto stamp = [&]() {
    if (kTune && p.dbg && blockIdx.x == 0 && threadIdx.x == 0) p.dbg[dbg_n++] = clock64();
  };
  stamp();
  timeline_mark(p.tl, p.tl_id, false);
  const RowTable* tab = p.tab;   // written before this pass started: safe to read ahead of the predecessor
  const int n_rows = tab->n_rows;
  const int HQ = p.n_q_heads * D;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int sub = lane / LPP, dl = lane % LPP;  // which position of the warp's group, which 8-dim slice
  const int total = tab->attn_items * p.n_kv_heads;
  bool waited = false;

  for (int item = blockIdx.x; item < total; item += gridDim.x) {
    const int kvh = item % p.n_kv_heads;
    const int rc = item / p.n_kv_heads;
    int row = 0;
    while (row + 1 < n_rows && tab->chunk_start[row + 1] <= rc) ++row;
    const int chunk = rc - tab->chunk_start[row];
    const int n_chunks = tab->chunk_start[row + 1] - tab->chunk_start[row];
    const int n_canon = tab->n_canon[row];
    const int p0 = chunk * ATT_CHUNK;
    const int n_can_here = min(ATT_CHUNK, n_canon - p0);
    const int n_spec = (chunk == n_chunks - 1) ? tab->n_spec[row] : 0;
    const int n_here = n_can_here + n_spec;
    // positions below n_safe were cached by earlier passes; the others are written by this pass's QKV kernel
    const int n_safe_can = min(n_can_here, max(0, tab->n_safe[row] - p0));
    const int n_safe = (n_spec > 0) ? n_can_here + n_spec - 1 : n_safe_can;

    const size_t plane = (size_t)(tab->r[row] - 1) * p.kv_plane_stride;
    const size_t headbase = (size_t)(tab->seq[row] * p.n_kv_heads + kvh) * p.slots * D;
    const __nv_bfloat16* Kb = p.kv + plane + headbase;
    const __nv_bfloat16* Vb = p.kv + plane + p.kv_sel_stride + headbase;

    auto slot_of = [&](int jpos) -> int { return jpos < n_can_here ? p0 + jpos : tab->spec_slot[row][jpos - n_can_here]; };
    uint4 kreg[ROUNDS], vreg[ROUNDS];
    auto load_kv = [&](int lo, int hi) {
#pragma unroll
      for (int rd = 0; rd < ROUNDS; ++rd) {
        const int jpos = rd * PPR + warp * PPW + sub;
        if (jpos >= lo && jpos < hi) {
          const size_t off = (size_t)slot_of(jpos) * D + dl * 8;
          kreg[rd] = *reinterpret_cast<const uint4*>(Kb + off);
          vreg[rd] = *reinterpret_cast<const uint4*>(Vb + off);
        }
      }
    };
#pragma unroll
    for (int rd = 0; rd < ROUNDS; ++rd) kreg[rd] = vreg[rd] = make_uint4(0, 0, 0, 0);
    stamp();
    load_kv(0, n_safe);
    stamp();
    if (!waited) {
      pdl_launch_dependents();
      pdl_wait();
      waited = true;
      timeline_mark(p.tl, p.tl_id + 256, false);
    }
    stamp();
    load_kv(n_safe, n_here);

    float q[G][8];
#pragma unroll
    for (int gq = 0; gq < G; ++gq) {
      const float4* qp =
          reinterpret_cast<const float4*>(p.qbuf + (size_t)row * p.n_q_heads * D + (size_t)(kvh * G + gq) * D + dl * 8);
      float4 a = qp[0], b = qp[1];
      q[gq][0] = a.x, q[gq][1] = a.y, q[gq][2] = a.z, q[gq][3] = a.w;
      q[gq][4] = b.x, q[gq][5] = b.y, q[gq][6] = b.z, q[gq][7] = b.w;
    }
    __syncthreads();  // shared buffers of the previous item are free
    stamp();

    // ---- scores ------------------------------------------------------------------------------------
#pragma unroll
    for (int rd = 0; rd < ROUNDS; ++rd) {
      const int jpos = rd * PPR + warp * PPW + sub;
      const unsigned w[4] = {kreg[rd].x, kreg[rd].y, kreg[rd].z, kreg[rd].w};
      float kf[8];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        kf[2 * i] = __uint_as_float(w[i] << 16);
        kf[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u);
      }
#pragma unroll
      for (int gq = 0; gq < G; ++gq) {
        float s = 0.f;
#pragma unroll
        for (int i = 0; i < 8; ++i) s = fmaf(q[gq][i], kf[i], s);
#pragma unroll
        for (int o = LPP / 2; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (dl == 0) s_score[gq][jpos] = (jpos < n_here) ? s * p.scale : -INFINITY;
      }
    }
    __syncthreads();
    stamp();

    // ---- chunk softmax statistics (one warp per query head, round robin) ----------------------------
    for (int gq = warp; gq < G; gq += ATT_THREADS / 32) {
      float m = -INFINITY;
      for (int jj = lane; jj < ROUNDS * PPR; jj += 32) m = fmaxf(m, s_score[gq][jj]);
      m = warp_max(m);
      float l = 0.f;
      for (int jj = lane; jj < ROUNDS * PPR; jj += 32) {
        float e = (jj < n_here) ? expf(s_score[gq][jj] - m) : 0.f;
        s_score[gq][jj] = e;
        l += e;
      }
      l = warp_sum(l);
      if (lane == 0) s_stat[gq][0] = m, s_stat[gq][1] = l;
    }
    __syncthreads();
    stamp();

    // ---- weighted values ----------------------------------------------------------------------------
    float o[G][8];
#pragma unroll
    for (int gq = 0; gq < G; ++gq)
#pragma unroll
      for (int i = 0; i < 8; ++i) o[gq][i] = 0.f;
#pragma unroll
    for (int rd = 0; rd < ROUNDS; ++rd) {
      const int jpos = rd * PPR + warp * PPW + sub;
      const unsigned w[4] = {vreg[rd].x, vreg[rd].y, vreg[rd].z, vreg[rd].w};
      float vf[8];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        vf[2 * i] = __uint_as_float(w[i] << 16);
        vf[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u);
      }
#pragma unroll
      for (int gq = 0; gq < G; ++gq) {
        float pw = s_score[gq][jpos];
#pragma unroll
        for (int i = 0; i < 8; ++i) o[gq][i] = fmaf(pw, vf[i], o[gq][i]);
      }
    }
    // fold the PPW position groups of the warp, then the warps, in fixed order
#pragma unroll
    for (int gq = 0; gq < G; ++gq)
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        float v = o[gq][i];
#pragma unroll
        for (int off = LPP; off < 32; off <<= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
        if (sub == 0) s_red[warp][gq][dl * 8 + i] = v;
      }
    __syncthreads();
    stamp();

    const int pair = row * p.n_kv_heads + kvh;
    float* mypart = p.part + ((size_t)pair * p.max_chunks + chunk) * G * PSTRIDE;
    if (n_chunks == 1) {
      for (int idx = tid; idx < G * D; idx += ATT_THREADS) {
        int gq = idx / D, dd = idx % D;
        float v = 0.f;
#pragma unroll
        for (int w2 = 0; w2 < ATT_THREADS / 32; ++w2) v += s_red[w2][gq][dd];
        store_split(p.aplanes + (size_t)row * 3 * HQ, HQ, (kvh * G + gq) * D + dd, v / s_stat[gq][1]);
      }
      continue;
    }
    for (int idx = tid; idx < G * D; idx += ATT_THREADS) {
      int gq = idx / D, dd = idx % D;
      float v = 0.f;
#pragma unroll
      for (int w2 = 0; w2 < ATT_THREADS / 32; ++w2) v += s_red[w2][gq][dd];
      __stcg(mypart + gq * PSTRIDE + dd, v);
    }
    if (tid < G) __stcg(mypart + tid * PSTRIDE + D, s_stat[tid][0]), __stcg(mypart + tid * PSTRIDE + D + 1, s_stat[tid][1]);
    __syncthreads();
    if (tid == 0) {
      __threadfence();
      int old = atomicAdd(p.counters + pair, 1);
      s_last = (old == n_chunks - 1);
      __threadfence();
    }
    __syncthreads();
    stamp();
    if (s_last) {  // combine the chunks in ascending order
      const float* base = p.part + (size_t)pair * p.max_chunks * G * PSTRIDE;
      for (int idx = tid; idx < G * D; idx += ATT_THREADS) {
        int gq = idx / D, dd = idx % D;
        float m = -INFINITY;
        for (int c0 = 0; c0 < n_chunks; c0 += 8) {
          float mm[8];
#pragma unroll
          for (int u = 0; u < 8; ++u) mm[u] = (c0 + u < n_chunks) ? __ldcg(base + ((size_t)(c0 + u) * G + gq) * PSTRIDE + D) : -INFINITY;
#pragma unroll
          for (int u = 0; u < 8; ++u) m = fmaxf(m, mm[u]);
        }
        float l = 0.f, acc = 0.f;
        for (int c0 = 0; c0 < n_chunks; c0 += 8) {
          float mc[8], lc[8], oc[8];
#pragma unroll
          for (int u = 0; u < 8; ++u) {
            const bool ok = c0 + u < n_chunks;
            const float* pc = base + ((size_t)(ok ? c0 + u : 0) * G + gq) * PSTRIDE;
            mc[u] = ok ? __ldcg(pc + D) : -INFINITY;
            lc[u] = ok ? __ldcg(pc + D + 1) : 0.f;
            oc[u] = ok ? __ldcg(pc + dd) : 0.f;
          }
#pragma unroll
          for (int u = 0; u < 8; ++u) {
            float wgt = expf(mc[u] - m);
            l = fmaf(lc[u], wgt, l);
            acc = fmaf(oc[u], wgt, acc);
          }
        }
        store_split(p.aplanes + (size_t)row * 3 * HQ, HQ, (kvh * G + gq) * D + dd, acc / l);
      }
      if (tid == 0) p.counters[pair] = 0;
    }
    stamp();
  }
  if (!waited) {
    pdl_launch_dependents();
    pdl_wait();
  }
  timeline_mark(p.tl, p.tl_id, true);
}

// ======================= decode attention on the tensor cores, one warp per item =====================================
// A work item is a run of consecutive chunks of one (row, kv head), cut as att_run_len says (a function of the row's own
// context); ONE warp streams it in tiles of 16 keys and keeps the running softmax, so nothing is folded across warps and no block
// barrier is met.  A CTA per item on the CUDA cores spends some 40 warp instructions on a key and 400 per item and warp; with many
// rows of short contexts that, not the stream, bounds it.  Here a tile is one mma.sync per 16 dims for the scores and one per 16
// dims for the values: K rows (V columns, by transposing ldmatrix) are the 16-row A operand, the query (the softmax weights) the
// columns - for G = 1 its three exact bf16 planes as columns 0 .. 2, for G = 4 the heads as columns 0 .. 3 with the planes one
// after the other into the same accumulator.  Every warp owns a ring of two tiles in shared memory, filled by its own cp.async
// across items; rows are swizzled in 16-byte pieces (ldmatrix without bank conflicts).
// A lone warp takes 1200 cycles per tile (310 issue the copies, 850 are the chain scores - softmax - values) and 4000 to 8000 per
// item around them, so what counts is that all items are resident at once: 12 warps per SM with tiles of 16 keys beat 6 with
// tiles of 32 [48 rows x 510 positions: 25.7 / 42.1 us] and 8 with three tiles each; deeper rings for few items change nothing.
// Alone, one CTA per run (CUDA cores) -> this kernel: 40 rows x 536 positions 61 -> 43 us, 24 rows 39 -> 23, 48 rows x 446
// 64 -> 26, 40 rows x 86 22 -> 12, 28 rows x 1036 69 -> 42, 14 rows x 8400 179 -> 154 us (6.25 TB/s).
template <int D, int G>
struct AtwCfg {
  static constexpr int WARPS = 4, STAGES = 2, CTAS = 3;  // CTAS: per SM
  static constexpr int ROWB = D * 2, KEYS = 16, TILE = KEYS * ROWB;  // bytes of a key row; keys of a tile and their bytes (values the same)
  static constexpr int QBYTES = G * D * 4;                 // an item's queries
  static constexpr int SMEM_BYTES = WARPS * STAGES * (2 * TILE + QBYTES);
};

__device__ __forceinline__ void att_ldsm4(unsigned (&r)[4], unsigned addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
__device__ __forceinline__ void att_ldsm4_t(unsigned (&r)[4], unsigned addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
__device__ __forceinline__ void att_mma(float (&c)[4], const unsigned (&a)[4], unsigned b0, unsigned b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
               : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
template <int D, int G>
__global__ void __launch_bounds__(AtwCfg<D, G>::WARPS * 32) attn_warp_kernel(const __grid_constant__ AttnParams p) {
  using C = AtwCfg<D, G>;
  static_assert(G == 1 || G == 4, "query heads per kv head");
  constexpr int PSTRIDE = D + 2, KS = D / 16, PCS = D / 8, NP = G == 1 ? 1 : 3;  // NP: column sets of a k-step (G = 1: planes are columns)
  constexpr int LI = C::KEYS * PCS / 32, RPI = 32 / PCS, SW = 8 / RPI;  // copies of keys per lane and tile, rows a copy of the warp covers, their swizzles
  extern __shared__ __align__(128) unsigned char atw_smem[];
  const RowTable* tab = p.tab;  // written before this pass started: safe to read ahead of the predecessor
  const int n_rows = tab->n_rows, HQ = p.n_q_heads * D;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int total = tab->attn_items * p.n_kv_heads, n_warps = gridDim.x * C::WARPS, first = warp * gridDim.x + blockIdx.x;  // (few items: one per SM first)
  const unsigned ring = (unsigned)__cvta_generic_to_shared(atw_smem) + warp * C::STAGES * 2 * C::TILE;
  float* const qring = reinterpret_cast<float*>(atw_smem + C::WARPS * C::STAGES * 2 * C::TILE) + warp * C::STAGES * (G * D);
  auto piece = [](int row, int c) { return (unsigned)(row * C::ROWB + ((c ^ (row & 7)) << 4)); };
  // this lane's row address of the fragment loads (dims 0 .. 15; the piece of a later k-step is two on: an XOR, the tiles being aligned)
  const unsigned k_lane = piece(lane & 15, lane >> 4), v_lane = piece((lane & 7) + ((lane >> 4) << 3), (lane >> 3) & 1);
  unsigned l_dst[SW];
#pragma unroll
  for (int i = 0; i < SW; ++i) l_dst[i] = (lane / PCS) * C::ROWB + (((lane % PCS) ^ ((lane / PCS + i * RPI) & 7)) << 4);

  // an item's keys: n_can committed ones from position p0 on, then (last run of the row) the speculative slots
  auto locate = [&](int item, int& row, int& kvh, int& run, int& p0, int& n_can, int& n_keys) {
    const int rr = item / p.n_kv_heads;
    kvh = item - rr * p.n_kv_heads;
    row = -1;  // the row whose items contain rr: as many rows start at or before it (one round trip to the table, not a search's five)
    for (int b = 0; b < n_rows; b += 32) row += __popc(__ballot_sync(0xffffffffu, b + lane < n_rows && tab->chunk_start[b + lane] <= rr));
    run = rr - tab->chunk_start[row];
    const int nc = tab->n_canon[row], len = att_run_len(nc, tab->att_mode) * ATT_CHUNK;
    p0 = run * len;
    n_can = min(len, nc - p0);
    n_keys = n_can + (p0 + len >= nc ? tab->n_spec[row] : 0);
  };
  // ---- ring, issue side: tiles of this warp's items in order, running ahead across items ----------------------------------
  int i_item = first, i_row = 0, i_p0 = 0, i_can = 0, i_keys = 0, i_j = 0;
  const __nv_bfloat16* i_kb = p.kv;
  auto i_setup = [&]() {
    int kvh, run;
    locate(i_item, i_row, kvh, run, i_p0, i_can, i_keys);
    i_kb = p.kv + (size_t)(tab->r[i_row] - 1) * p.kv_plane_stride + (size_t)(tab->seq[i_row] * p.n_kv_heads + kvh) * p.slots * D;
    i_j = 0;
  };
  if (i_item < total) i_setup();
  unsigned i_st = 0, c_st = 0;
  int i_q = 0, c_q = 0;        // query slot of the item being issued / consumed
  bool queries = false;        // the queries exist (they are this pass's: not ahead of the dependency wait)
  auto issue_q = [&](int row, int kvh, int qs) {
    for (int i = lane; i < G * D / 4; i += 32)
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(qring + qs * (G * D) + i * 4)),
                   "l"(p.qbuf + (size_t)row * HQ + (size_t)kvh * G * D + i * 4)
                   : "memory");
  };
  auto issue = [&]() {
    if (i_item < total) {
      if (i_j == 0 && queries) issue_q(i_row, i_item % p.n_kv_heads, i_q);
      if (i_j + C::KEYS <= i_can) {  // a full tile of committed keys: constant strides from this lane's first piece
        const __nv_bfloat16* k0 = i_kb + (size_t)(i_p0 + i_j) * D + lane * 8;
        const __nv_bfloat16* v0 = k0 + p.kv_sel_stride;
#pragma unroll
        for (int i = 0; i < LI; ++i) {
          const unsigned dst = ring + i_st + i * RPI * C::ROWB + l_dst[i % SW];
          asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(k0 + i * 256) : "memory");
          asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + C::TILE), "l"(v0 + i * 256) : "memory");
        }
      } else {
#pragma unroll 1
        for (int i = 0; i < LI; ++i) {
          const int r = lane / PCS + i * RPI, c = lane % PCS, j = i_j + r;
          const bool live = j < i_keys;  // keys beyond the item: zeros
          const int slot = j < i_can ? i_p0 + j : (live ? tab->spec_slot[i_row][j - i_can] : 0);
          const __nv_bfloat16* src = i_kb + (size_t)slot * D + c * 8;
          const unsigned dst = ring + i_st + piece(r, c);
          const int n = live ? 16 : 0;
          asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(n) : "memory");
          asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst + C::TILE), "l"(src + p.kv_sel_stride), "r"(n) : "memory");
        }
      }
      i_j += C::KEYS;
      if (i_j >= i_keys) {
        i_item += n_warps;
        if (++i_q == C::STAGES) i_q = 0;
        if (i_item < total) i_setup();
      }
    }
    i_st += 2 * C::TILE;
    if (i_st == C::STAGES * 2 * C::TILE) i_st = 0;
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  {
    int issued = 0;
    // tiles whose keys were all cached by earlier passes are requested ahead of the predecessor's completion (committed
    // positions below n_safe, and every speculative slot but the row's own; the others are written by this pass's QKV kernel)
    while (issued < C::STAGES - 1 && i_item < total) {
      const int n_safe = i_keys > i_can ? i_keys - 1 : min(i_can, max(0, tab->n_safe[i_row] - i_p0));
      if (min(i_j + C::KEYS, i_keys) > n_safe) break;
      issue(), ++issued;
    }
    pdl_launch_dependents();
    pdl_wait();
    queries = true;
    if (issued > 0) {  // the queries of the items whose tiles went out above
      int qs = 0;
      for (int it = first; it < total && (it < i_item || (it == i_item && i_j > 0)); it += n_warps, ++qs) {
        int row, kvh, run, p0, n_can, n_keys;
        locate(it, row, kvh, run, p0, n_can, n_keys);
        issue_q(row, kvh, qs);
      }
      asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
    }
    for (; issued < C::STAGES - 1; ++issued) issue();
  }
  // A finished item's arrival is announced one item later, when its stores have long landed; the warp that announces the last
  // run of a (row, kv head) folds the runs in ascending order, D / 32 dims per lane
  int pend_row = -1, pend_kvh = 0;
  auto arrive = [&]() {
    const int row = pend_row, kvh = pend_kvh, pair = row * p.n_kv_heads + kvh, n_runs = tab->chunk_start[row + 1] - tab->chunk_start[row];
    __threadfence();
    __syncwarp();
    int old = 0;
    if (lane == 0) old = atomicAdd(p.counters + pair, 1);
    old = __shfl_sync(0xffffffffu, old, 0);
    if (old != n_runs - 1) return;
    __threadfence();
    constexpr int DPV = D / 32;
    for (int gq = 0; gq < G; ++gq) {
      const float* base = p.part + ((size_t)pair * p.max_chunks * G + gq) * PSTRIDE;
      constexpr size_t RS = (size_t)G * PSTRIDE;
      float mx = -INFINITY, ll = 0.f, acc[DPV];
#pragma unroll
      for (int d = 0; d < DPV; ++d) acc[d] = 0.f;
      for (int c0 = 0; c0 < n_runs; c0 += 8) {
        float mc[8], lc[8];
        float2 oc[8][DPV / 2];  // (a partial's D + 2 floats keep 8-byte alignment only)
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const bool live = c0 + u < n_runs;
          const float* pc = base + (size_t)(live ? c0 + u : 0) * RS;
          mc[u] = live ? __ldcg(pc + D) : -INFINITY, lc[u] = live ? __ldcg(pc + D + 1) : 0.f;
#pragma unroll
          for (int d = 0; d < DPV / 2; ++d) oc[u][d] = live ? __ldcg(reinterpret_cast<const float2*>(pc + lane * DPV) + d) : make_float2(0.f, 0.f);
        }
        float mn = mx;
#pragma unroll
        for (int u = 0; u < 8; ++u) mn = fmaxf(mn, mc[u]);
        const float wa = mx == -INFINITY ? 0.f : expf(mx - mn);
        mx = mn, ll *= wa;
#pragma unroll
        for (int d = 0; d < DPV; ++d) acc[d] *= wa;
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const float wgt = mc[u] == -INFINITY ? 0.f : expf(mc[u] - mx);
          ll = fmaf(lc[u], wgt, ll);
#pragma unroll
          for (int d = 0; d < DPV / 2; ++d) acc[2 * d] = fmaf(oc[u][d].x, wgt, acc[2 * d]), acc[2 * d + 1] = fmaf(oc[u][d].y, wgt, acc[2 * d + 1]);
        }
      }
#pragma unroll
      for (int d = 0; d < DPV; d += 2) store_split2(p.aplanes + (size_t)row * 3 * HQ, HQ, (kvh * G + gq) * D + lane * DPV + d, acc[d] / ll, acc[d + 1] / ll);
    }
    if (lane == 0) p.counters[pair] = 0;
  };

  for (int item = first; item < total; item += n_warps) {
    int row, kvh, run, p0, n_can, n_keys;
    locate(item, row, kvh, run, p0, n_can, n_keys);
    constexpr int NH = G == 1 ? 1 : 2;  // heads a lane keeps the softmax state of (G = 4: heads 2 t, 2 t + 1 in lanes t < 2)
    float m[NH], l[NH], o[KS][4];
#pragma unroll
    for (int h = 0; h < NH; ++h) m[h] = -INFINITY, l[h] = 0.f;
#pragma unroll
    for (int ks = 0; ks < KS; ++ks)
#pragma unroll
      for (int i = 0; i < 4; ++i) o[ks][i] = 0.f;

    unsigned qf[KS][NP][2];
    for (int j0 = 0; j0 < n_keys; j0 += C::KEYS) {
      issue();
      asm volatile("cp.async.wait_group %0;" ::"n"(C::STAGES - 1) : "memory");
      __syncwarp();
      if (j0 == 0) {  // the queries came with the first tile: dims 16 ks + 2 t, + 1 (first register) and + 8, + 9 (second) of column g
#pragma unroll
        for (int ks = 0; ks < KS; ++ks) {
          const bool live = G == 1 ? g < 3 : g < 4;
          float2 a = make_float2(0.f, 0.f), b = a;
          if (live) {
            const float* qp = qring + c_q * (G * D) + (G == 1 ? 0 : g) * D + 16 * ks + 2 * t;
            a = *reinterpret_cast<const float2*>(qp), b = *reinterpret_cast<const float2*>(qp + 8);
          }
          unsigned pa[3], pb[3];
          split3_pair(a.x, a.y, pa), split3_pair(b.x, b.y, pb);
          if constexpr (G == 1) {
            qf[ks][0][0] = g == 0 ? pa[0] : g == 1 ? pa[1] : pa[2];
            qf[ks][0][1] = g == 0 ? pb[0] : g == 1 ? pb[1] : pb[2];
          } else {
#pragma unroll
            for (int s = 0; s < 3; ++s) qf[ks][s][0] = pa[s], qf[ks][s][1] = pb[s];
          }
        }
        if (++c_q == C::STAGES) c_q = 0;
      }
      const unsigned kt = ring + c_st, vt = kt + C::TILE;
      // ---- scores of keys g and g + 8 of every row tile ----
      unsigned fr[KS][4];  // every fragment is requested before the first is used: a load waited for is 30 cycles of a lone warp's chain
#pragma unroll
      for (int ks = 0; ks < KS; ++ks) att_ldsm4(fr[ks], (kt + k_lane) ^ (ks << 5));
      float sc[4];
      {
        float c[4][4];  // four chains over the k-steps
#pragma unroll
        for (int x = 0; x < 4; ++x)
#pragma unroll
          for (int i = 0; i < 4; ++i) c[x][i] = 0.f;
#pragma unroll
        for (int ks = 0; ks < KS; ++ks)
#pragma unroll
          for (int s = 0; s < NP; ++s) att_mma(c[ks & 3], fr[ks], qf[ks][s][0], qf[ks][s][1]);
#pragma unroll
        for (int i = 0; i < 4; ++i) sc[i] = (c[0][i] + c[1][i]) + (c[2][i] + c[3][i]);
      }
#pragma unroll
      for (int ks = 0; ks < KS; ++ks)  // (the value columns arrive under the softmax)
        att_ldsm4_t(fr[ks], (vt + v_lane) ^ (ks << 5));
      float e0[NH], e1[NH], wa[NH];  // (key g, key g + 8) of this lane's heads: score, then softmax weight
      if constexpr (G == 1) {  // columns 0, 1 (planes hi, mid) sit in lane t = 0, column 2 (lo) in t = 1; every lane takes the sum
        const int b = lane & ~3;
        e0[0] = __shfl_sync(0xffffffffu, sc[0], b) + (__shfl_sync(0xffffffffu, sc[1], b) + __shfl_sync(0xffffffffu, sc[0], b + 1));
        e1[0] = __shfl_sync(0xffffffffu, sc[2], b) + (__shfl_sync(0xffffffffu, sc[3], b) + __shfl_sync(0xffffffffu, sc[2], b + 1));
      } else {
#pragma unroll
        for (int h = 0; h < 2; ++h) e0[h] = sc[h], e1[h] = sc[2 + h];
      }
      bool moved = false;
#pragma unroll
      for (int h = 0; h < NH; ++h) {  // running softmax
        float mx = -INFINITY;
        e0[h] = j0 + g < n_keys ? e0[h] * p.scale : -INFINITY;
        e1[h] = j0 + g + 8 < n_keys ? e1[h] * p.scale : -INFINITY;
        mx = fmaxf(mx, fmaxf(e0[h], e1[h]));
#pragma unroll
        for (int off = 4; off < 32; off <<= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, off));
        mx = fmaxf(mx, m[h]);  // (finite: every tile holds a key)
        wa[h] = m[h] == -INFINITY ? 0.f : expf(m[h] - mx);
        moved |= mx != m[h];
        m[h] = mx;
        float sum = 0.f;
        e0[h] = expf(e0[h] - mx), e1[h] = expf(e1[h] - mx);
        sum += e0[h] + e1[h];
        l[h] = fmaf(l[h], wa[h], sum);  // (this lane's keys; summed over the lanes when the run is done)
      }
      if (G == 1 ? moved : __any_sync(0xffffffffu, moved)) {
#pragma unroll
        for (int ks = 0; ks < KS; ++ks)
#pragma unroll
          for (int i = 0; i < 4; ++i) o[ks][i] *= wa[G == 1 ? 0 : (i & 1)];
      }
      // ---- softmax weights as columns: keys 2 t, 2 t + 1 (first register), + 8, + 9 (second) of column g ----
      unsigned pf[NP][2];
      float a[2], b[2];
      const int l0 = 8 * t, l1 = 8 * t + 4;  // lanes (key 2 t, .) and (key 2 t + 1, .)
      if constexpr (G == 1) {
        a[0] = __shfl_sync(0xffffffffu, e0[0], l0), a[1] = __shfl_sync(0xffffffffu, e0[0], l1);
        b[0] = __shfl_sync(0xffffffffu, e1[0], l0), b[1] = __shfl_sync(0xffffffffu, e1[0], l1);
      } else {  // column g = head g: state in lane t = g / 2, register g & 1
        const int src = (g >> 1) & 1;
#pragma unroll
        for (int x = 0; x < 2; ++x) {
          const int from = (x ? l1 : l0) + src;
          const float u0 = __shfl_sync(0xffffffffu, e0[0], from), u1 = __shfl_sync(0xffffffffu, e0[NH - 1], from);
          const float w0 = __shfl_sync(0xffffffffu, e1[0], from), w1 = __shfl_sync(0xffffffffu, e1[NH - 1], from);
          a[x] = g >= 4 ? 0.f : (g & 1) ? u1 : u0, b[x] = g >= 4 ? 0.f : (g & 1) ? w1 : w0;
        }
      }
      unsigned pa[3], pb[3];
      split3_pair(a[0], a[1], pa), split3_pair(b[0], b[1], pb);
      if constexpr (G == 1) {
        pf[0][0] = g == 0 ? pa[0] : g == 1 ? pa[1] : g == 2 ? pa[2] : 0u;
        pf[0][1] = g == 0 ? pb[0] : g == 1 ? pb[1] : g == 2 ? pb[2] : 0u;
      } else {
#pragma unroll
        for (int s = 0; s < 3; ++s) pf[s][0] = pa[s], pf[s][1] = pb[s];
      }
#pragma unroll
      for (int s = 0; s < NP; ++s)
#pragma unroll
        for (int ks = 0; ks < KS; ++ks) att_mma(o[ks], fr[ks], pf[s][0], pf[s][1]);  // dims 16 ks .. + 15
      __syncwarp();  // the tile may be overwritten
      c_st += 2 * C::TILE;
      if (c_st == C::STAGES * 2 * C::TILE) c_st = 0;
    }

    // ---- the run is done: dims 16 ks + g and + 8 of this lane's heads ----
#pragma unroll
    for (int h = 0; h < NH; ++h)
#pragma unroll
      for (int off = 4; off < 32; off <<= 1) l[h] += __shfl_xor_sync(0xffffffffu, l[h], off);
    const int pair = row * p.n_kv_heads + kvh, n_runs = tab->chunk_start[row + 1] - tab->chunk_start[row];
    float* mypart = p.part + ((size_t)pair * p.max_chunks + run) * G * PSTRIDE;
    auto out = [&](int gq, int dd, float v, float mass) {
      if (n_runs == 1) store_split(p.aplanes + (size_t)row * 3 * HQ, HQ, (kvh * G + gq) * D + dd, v / mass);
      else __stcg(mypart + gq * PSTRIDE + dd, v);
    };
#pragma unroll
    for (int ks = 0; ks < KS; ++ks) {
      if constexpr (G == 1) {
        const float lo0 = __shfl_sync(0xffffffffu, o[ks][0], (lane & ~3) + 1), lo1 = __shfl_sync(0xffffffffu, o[ks][2], (lane & ~3) + 1);
        if (t == 0) out(0, 16 * ks + g, o[ks][0] + (o[ks][1] + lo0), l[0]), out(0, 16 * ks + g + 8, o[ks][2] + (o[ks][3] + lo1), l[0]);
      } else if (t < 2) {
#pragma unroll
        for (int h = 0; h < NH; ++h) out(2 * t + h, 16 * ks + g, o[ks][h], l[h]), out(2 * t + h, 16 * ks + g + 8, o[ks][2 + h], l[h]);
      }
    }
    if (n_runs == 1) continue;
    if (g == 0 && t < (G == 1 ? 1 : 2)) {
#pragma unroll
      for (int h = 0; h < NH; ++h) __stcg(mypart + (NH * t + h) * PSTRIDE + D, m[h]), __stcg(mypart + (NH * t + h) * PSTRIDE + D + 1, l[h]);
    }
    if (pend_row >= 0) arrive();
    pend_row = row, pend_kvh = kvh;
  }
  if (pend_row >= 0) arrive();
  asm volatile("cp.async.wait_group 0;" ::: "memory");  // (only empty groups are left)
}

// ======================= prefill attention: the rows of a pass share every key / value chunk ========================
// A prefill pass carries consecutive prompt positions p0 .. p0 + n - 1 of one sequence at one recurrence, so all its rows
// read the same cached keys and values (row i up to its own position).  A work item is (query head, block of 32 rows, run
// of chunks): a chunk's keys and values are brought into shared memory once for the block, and every row keeps a running
// softmax over the chunks of the run.  Runs are cut at fixed absolute positions - every chunk below position
// ATT_PF_SINGLE * 64 is a run of its own, beyond that runs of ATT_PF_RUN chunks - and a row's runs are folded in ascending
// order by a second kernel (attn_prefill_fold_kernel), so a row's result depends on its own prefix only, not on how the
// prompt was cut into passes.
constexpr int ATT_PF_SINGLE = 8;  // [measured per layer at 2048 / 4096 / 8192 positions, 64 rows: single chunks up to 8 and runs of 4
constexpr int ATT_PF_RUN = 4;     //  beyond: 43 / 68 / 106 us; up to 16: 47 / 66 / 120 us; up to 40: 51 / 78 / 133 us; runs of 8: slower]
__host__ __device__ inline int att_pf_run_of_chunk(int c) { return c < ATT_PF_SINGLE ? c : ATT_PF_SINGLE + (c - ATT_PF_SINGLE) / ATT_PF_RUN; }
__host__ __device__ inline int att_pf_run_first_chunk(int run) {
  return run < ATT_PF_SINGLE ? run : ATT_PF_SINGLE + (run - ATT_PF_SINGLE) * ATT_PF_RUN;
}
constexpr int ATT_PF_ROWS = 64;  // rows of a pass at most (one group of token columns)

// Scores and weighted values of a (32 rows x 64 keys) tile are mma.sync.m16n8k16 contractions (bf16 x bf16 -> fp32).  Keys
// and values are bf16 already; the fp32 queries and the fp32 softmax weights are split exactly into three bf16 planes
// (hi + mid + lo), one accumulator chain per plane, folded hi + (mid + lo) - the arithmetic of the GEMM kernels, so every
// product is exact and a row's result depends on its own operands only (not on its place in the tile, nor on the other
// rows).  (The same tiles as fp32 FMAs in registers took 29 us per layer at 512 positions and 211 us at 8192 against 18 us
// and 134 us here.)
template <int D>
struct AtmCfg {
  static constexpr int IR = 32;                 // rows per item: two 16-row MMA tiles
  static constexpr int QS = D + 8;              // bf16 per row of a query plane (the pad keeps fragment loads off each other's banks)
  static constexpr int KS = D + 8;              // bf16 per key / value row
  static constexpr int PS = ATT_CHUNK + 8;      // bf16 per row of a softmax-weight plane
  static constexpr int SS = ATT_CHUNK + 1;      // floats per score row
  static constexpr int Q_OFF = 0;                                   // [3][IR][QS] bf16
  static constexpr int K_OFF = Q_OFF + 3 * IR * QS * 2;             // [64][KS] bf16
  static constexpr int V_OFF = K_OFF + ATT_CHUNK * KS * 2;          // [64][KS] bf16
  static constexpr int P_OFF = V_OFF + ATT_CHUNK * KS * 2;          // [3][IR][PS] bf16
  static constexpr int S_OFF = P_OFF + 3 * IR * PS * 2;             // [IR][SS] fp32
  static constexpr int ST_OFF = S_OFF + IR * SS * 4;                // [IR][4] fp32
  static constexpr int SMEM_BYTES = ST_OFF + IR * 4 * 4;
};

template <int D>
__global__ void __launch_bounds__(ATT_THREADS, 2) attn_prefill_mma_kernel(const __grid_constant__ AttnParams p) {
  using C = AtmCfg<D>;
  constexpr int IR = C::IR, PSTRIDE = D + 2;
  constexpr int NTO = D / 32;  // 8-dim output tiles per warp (each warp: one 16-row tile x NTO column tiles)
  extern __shared__ __align__(16) unsigned char atm_smem[];
  __nv_bfloat16* s_q = reinterpret_cast<__nv_bfloat16*>(atm_smem + C::Q_OFF);
  __nv_bfloat16* s_k = reinterpret_cast<__nv_bfloat16*>(atm_smem + C::K_OFF);
  __nv_bfloat16* s_v = reinterpret_cast<__nv_bfloat16*>(atm_smem + C::V_OFF);
  __nv_bfloat16* s_p = reinterpret_cast<__nv_bfloat16*>(atm_smem + C::P_OFF);
  float* s_s = reinterpret_cast<float*>(atm_smem + C::S_OFF);
  float* s_st = reinterpret_cast<float*>(atm_smem + C::ST_OFF);  // [row][4]: running max, running mass, rescale of this chunk

  const RowTable* tab = p.tab;  // written before this pass started
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
  const int n_rows = min(tab->n_rows, ATT_PF_ROWS);
  pdl_launch_dependents();
  pdl_wait();  // the queries, and the keys / values of the pass's own positions, come from this pass's QKV kernel
  if (n_rows <= 0) return;
  const int p0 = tab->pos[0], seq = tab->seq[0];
  const int n_ctx = p0 + n_rows;                                   // keys 0 .. n_ctx - 1
  const int n_runs_all = att_pf_run_of_chunk((n_ctx - 1) / ATT_CHUNK) + 1;
  const int n_blocks = (n_rows + IR - 1) / IR;
  const int G = p.n_q_heads / p.n_kv_heads, HQ = p.n_q_heads * D;
  const size_t plane = (size_t)(tab->r[0] - 1) * p.kv_plane_stride;
  const int total = p.n_q_heads * n_blocks * n_runs_all;
  const int mt = warp & 1;   // this warp's 16-row tile
  const int wq = warp >> 1;  // ... and its quarter of the columns (keys of the score tile, dims of the output tile)

  for (int item = blockIdx.x; item < total; item += gridDim.x) {
    const int h = item % p.n_q_heads, rest = item / p.n_q_heads;
    const int blk = rest % n_blocks, run = rest / n_blocks;
    const int row0 = blk * IR, rows_here = min(IR, n_rows - row0);  // this item's rows of the pass
    const int kvh = h / G, gq = h - kvh * G;
    const int c_lo = att_pf_run_first_chunk(run);
    // keys beyond the block's last position are never visible to it: the run ends there
    const int c_hi = min(att_pf_run_first_chunk(run + 1), (p0 + row0 + rows_here - 1) / ATT_CHUNK + 1);
    if (c_lo >= c_hi) continue;  // (uniform over the CTA) none of the block's rows reaches this run
    const __nv_bfloat16* Kb = p.kv + plane + (size_t)(seq * p.n_kv_heads + kvh) * p.slots * D;
    const __nv_bfloat16* Vb = Kb + p.kv_sel_stride;
    __syncthreads();  // the previous item is done with the shared buffers
    // the block's queries for this head, split into three bf16 planes; rows the pass does not have are zeros
    for (int idx = tid; idx < IR * (D / 4); idx += ATT_THREADS) {
      const int lr = idx / (D / 4), d4 = idx - lr * (D / 4);
      float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
      if (lr < rows_here) v = *reinterpret_cast<const float4*>(p.qbuf + (size_t)(row0 + lr) * HQ + (size_t)h * D + d4 * 4);
      const float x[4] = {v.x, v.y, v.z, v.w};
      unsigned short hh[4], mm[4], ll[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) split3(x[i], hh[i], mm[i], ll[i]);
      __nv_bfloat16* q0 = s_q + lr * C::QS + d4 * 4;
      *reinterpret_cast<uint2*>(q0) = make_uint2(hh[0] | ((unsigned)hh[1] << 16), hh[2] | ((unsigned)hh[3] << 16));
      *reinterpret_cast<uint2*>(q0 + IR * C::QS) = make_uint2(mm[0] | ((unsigned)mm[1] << 16), mm[2] | ((unsigned)mm[3] << 16));
      *reinterpret_cast<uint2*>(q0 + 2 * IR * C::QS) = make_uint2(ll[0] | ((unsigned)ll[1] << 16), ll[2] | ((unsigned)ll[3] << 16));
    }
    if (tid < IR) s_st[tid * 4] = -INFINITY, s_st[tid * 4 + 1] = 0.f, s_st[tid * 4 + 2] = 1.f;
    float o[NTO][4];  // running weighted values: rows 16 mt + g (elements 0, 1) and + 8 (2, 3), dims 8 (wq NTO + j) + 2 t, + 1
#pragma unroll
    for (int j = 0; j < NTO; ++j)
#pragma unroll
      for (int i = 0; i < 4; ++i) o[j][i] = 0.f;

    for (int chunk = c_lo; chunk < c_hi; ++chunk) {
      const int k0 = chunk * ATT_CHUNK;
      const int n_keys = min(ATT_CHUNK, n_ctx - k0);  // keys of this chunk that exist (all of them written)
      if (chunk > c_lo) __syncthreads();               // the previous chunk's readers are done
      // ---- the chunk's keys and values, once for all rows of the block (missing keys: zeros) ----------------------
      for (int idx = tid; idx < ATT_CHUNK * (D / 8); idx += ATT_THREADS) {
        const int key = idx / (D / 8), pc = idx - key * (D / 8);
        const bool ok = key < n_keys;
        const size_t off = (size_t)(k0 + (ok ? key : 0)) * D + pc * 8;
        cp_async16_zfill(s_k + key * C::KS + pc * 8, Kb + off, ok);
        cp_async16_zfill(s_v + key * C::KS + pc * 8, Vb + off, ok);
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
      asm volatile("cp.async.wait_group 0;" ::: "memory");
      __syncthreads();
      // ---- scores: this warp's 16 rows x 16 keys (two 8-key tiles), three plane chains each --------------------------
      {
        float acc[3][2][4];
#pragma unroll
        for (int pl = 0; pl < 3; ++pl)
#pragma unroll
          for (int j = 0; j < 2; ++j)
#pragma unroll
            for (int i = 0; i < 4; ++i) acc[pl][j][i] = 0.f;
#pragma unroll 2
        for (int ks = 0; ks < D / 16; ++ks) {
          unsigned a[3][4];
#pragma unroll
          for (int pl = 0; pl < 3; ++pl) {
            const __nv_bfloat16* qa = s_q + (pl * IR + 16 * mt + g) * C::QS + 16 * ks + 2 * t;
            a[pl][0] = *reinterpret_cast<const unsigned*>(qa), a[pl][1] = *reinterpret_cast<const unsigned*>(qa + 8 * C::QS);
            a[pl][2] = *reinterpret_cast<const unsigned*>(qa + 8), a[pl][3] = *reinterpret_cast<const unsigned*>(qa + 8 * C::QS + 8);
          }
#pragma unroll
          for (int j = 0; j < 2; ++j) {
            const __nv_bfloat16* kb = s_k + (8 * (2 * wq + j) + g) * C::KS + 16 * ks + 2 * t;
            const unsigned b0 = *reinterpret_cast<const unsigned*>(kb), b1 = *reinterpret_cast<const unsigned*>(kb + 8);
#pragma unroll
            for (int pl = 0; pl < 3; ++pl) att_mma(acc[pl][j], a[pl], b0, b1);
          }
        }
#pragma unroll
        for (int j = 0; j < 2; ++j)
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const int lr = 16 * mt + g + (i >> 1) * 8, key = 8 * (2 * wq + j) + 2 * t + (i & 1);
            const float sv = acc[0][j][i] + (acc[1][j][i] + acc[2][j][i]);
            const bool ok = lr < rows_here && key < n_keys && k0 + key <= p0 + row0 + lr;  // causal
            s_s[lr * C::SS + key] = ok ? sv * p.scale : -INFINITY;
          }
      }
      __syncthreads();
      // ---- running softmax of every row: four threads per row, 16 keys each, folded in a fixed order; the weights go
      // to three bf16 planes for the second contraction -------------------------------------------------------------
      if (tid < 4 * IR) {
        const int lr = tid >> 2, part = tid & 3;
        const float* sr = s_s + lr * C::SS + part * 16;
        float m = -INFINITY;
#pragma unroll
        for (int jj = 0; jj < 16; ++jj) m = fmaxf(m, sr[jj]);
        m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 1));
        m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 2));
        const float m_old = s_st[lr * 4], l_old = s_st[lr * 4 + 1];
        const float m_new = fmaxf(m_old, m);
        float l = 0.f;
#pragma unroll
        for (int jj = 0; jj < 16; jj += 2) {
          const float e0 = (sr[jj] == -INFINITY) ? 0.f : expf(sr[jj] - m_new);
          const float e1 = (sr[jj + 1] == -INFINITY) ? 0.f : expf(sr[jj + 1] - m_new);
          l += e0;
          l += e1;
          unsigned short h0, m0, l0, h1, m1, l1;
          split3(e0, h0, m0, l0);
          split3(e1, h1, m1, l1);
          __nv_bfloat16* pp = s_p + lr * C::PS + part * 16 + jj;
          *reinterpret_cast<unsigned*>(pp) = h0 | ((unsigned)h1 << 16);
          *reinterpret_cast<unsigned*>(pp + IR * C::PS) = m0 | ((unsigned)m1 << 16);
          *reinterpret_cast<unsigned*>(pp + 2 * IR * C::PS) = l0 | ((unsigned)l1 << 16);
        }
        const float l1s = __shfl_xor_sync(0xffffffffu, l, 1);
        const float lp = (part & 1) ? l1s + l : l + l1s;       // (part 0 + part 1), (part 2 + part 3)
        const float l2s = __shfl_xor_sync(0xffffffffu, lp, 2);
        const float lc = (part & 2) ? l2s + lp : lp + l2s;     // lower pair first
        __syncwarp();
        if (part == 0) {
          const float wa = (m_old == -INFINITY) ? 0.f : expf(m_old - m_new);  // (a row that has seen no key yet: nothing to rescale)
          s_st[lr * 4] = m_new, s_st[lr * 4 + 1] = fmaf(l_old, wa, lc), s_st[lr * 4 + 2] = (m_new == -INFINITY) ? 1.f : wa;
        }
      }
      __syncthreads();
      // ---- weighted values: this warp's 16 rows x NTO tiles of 8 dims, keys in four steps of 16 ---------------------------
      {
        float acc[3][NTO][4];
#pragma unroll
        for (int pl = 0; pl < 3; ++pl)
#pragma unroll
          for (int j = 0; j < NTO; ++j)
#pragma unroll
            for (int i = 0; i < 4; ++i) acc[pl][j][i] = 0.f;
#pragma unroll
        for (int ks = 0; ks < ATT_CHUNK / 16; ++ks) {
          unsigned a[3][4];
#pragma unroll
          for (int pl = 0; pl < 3; ++pl) {
            const __nv_bfloat16* pa = s_p + (pl * IR + 16 * mt + g) * C::PS + 16 * ks + 2 * t;
            a[pl][0] = *reinterpret_cast<const unsigned*>(pa), a[pl][1] = *reinterpret_cast<const unsigned*>(pa + 8 * C::PS);
            a[pl][2] = *reinterpret_cast<const unsigned*>(pa + 8), a[pl][3] = *reinterpret_cast<const unsigned*>(pa + 8 * C::PS + 8);
          }
#pragma unroll
          for (int j = 0; j < NTO; ++j) {
            // B fragment of V[key][dim] (keys = the contraction index): transposing matrix load, lanes 0-15 name the key rows
            const unsigned addr = (unsigned)__cvta_generic_to_shared(s_v + (16 * ks + (lane & 15)) * C::KS + 8 * (wq * NTO + j));
            unsigned b0, b1;
            asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0,%1}, [%2];" : "=r"(b0), "=r"(b1) : "r"(addr));
#pragma unroll
            for (int pl = 0; pl < 3; ++pl) att_mma(acc[pl][j], a[pl], b0, b1);
          }
        }
        const float wa0 = s_st[(16 * mt + g) * 4 + 2], wa1 = s_st[(16 * mt + g + 8) * 4 + 2];
#pragma unroll
        for (int j = 0; j < NTO; ++j)
#pragma unroll
          for (int i = 0; i < 4; ++i)
            o[j][i] = fmaf(o[j][i], (i >> 1) ? wa1 : wa0, acc[0][j][i] + (acc[1][j][i] + acc[2][j][i]));
      }
    }
    __syncthreads();  // every thread has read the final state
    // ---- the run is done: rows with one run only are finished here, the others leave a partial for the fold -----------
#pragma unroll
    for (int hf = 0; hf < 2; ++hf) {
      const int lr = 16 * mt + g + 8 * hf, row = row0 + lr, pos = p0 + row;
      if (lr >= rows_here || c_lo * ATT_CHUNK > pos) continue;   // the row does not reach this run
      const int n_runs_row = att_pf_run_of_chunk(pos / ATT_CHUNK) + 1;
      const float m = s_st[lr * 4], l = s_st[lr * 4 + 1];
      float* mypart = p.part + (((size_t)(row * p.n_kv_heads + kvh) * p.max_chunks + run) * G + gq) * PSTRIDE;
#pragma unroll
      for (int j = 0; j < NTO; ++j)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const int dd = 8 * (wq * NTO + j) + 2 * t + e;
          const float v = o[j][2 * hf + e];
          if (n_runs_row == 1) store_split(p.aplanes + (size_t)row * 3 * HQ, HQ, h * D + dd, v / l);
          else __stcg(mypart + dd, v);
        }
      if (n_runs_row > 1 && wq == 0 && t == 0) __stcg(mypart + D, m), __stcg(mypart + D + 1, l);
    }
  }
}

// ... and the fold of a row's runs, in ascending order: one CTA per (row, query head), one lane per four dims.  A
// kernel of its own so that the folds of a pass (up to 64 rows x all heads x up to ATT_PF_SINGLE + max_ctx / 1024 runs)
// spread over the whole device instead of queuing in whichever CTA finished a head last.
template <int D>
__global__ void __launch_bounds__(D / 4) attn_prefill_fold_kernel(const __grid_constant__ AttnParams p) {
  constexpr int PSTRIDE = D + 2;
  const RowTable* tab = p.tab;
  const int row = blockIdx.x, h = blockIdx.y, tid = threadIdx.x;
  pdl_launch_dependents();
  pdl_wait();
  if (row >= min(tab->n_rows, ATT_PF_ROWS)) return;
  const int n_runs = att_pf_run_of_chunk(tab->pos[row] / ATT_CHUNK) + 1;
  if (n_runs == 1) return;  // finished by the attention kernel itself
  const int G = p.n_q_heads / p.n_kv_heads, HQ = p.n_q_heads * D, kvh = h / G, gq = h - kvh * G;
  const float* base = p.part + ((size_t)(row * p.n_kv_heads + kvh) * p.max_chunks * G + gq) * PSTRIDE;
  const size_t rstride = (size_t)G * PSTRIDE;
  float m = -INFINITY;
  for (int c0 = 0; c0 < n_runs; c0 += 8) {
    float mm[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) mm[u] = (c0 + u < n_runs) ? __ldcg(base + (size_t)(c0 + u) * rstride + D) : -INFINITY;
#pragma unroll
    for (int u = 0; u < 8; ++u) m = fmaxf(m, mm[u]);
  }
  float l = 0.f, acc[4] = {0.f, 0.f, 0.f, 0.f};
  for (int c0 = 0; c0 < n_runs; c0 += 8) {
    float mc[8], lc[8];
    float2 oa[8], ob[8];  // (a partial's D + 2 floats keep 8-byte alignment only)
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const bool ok = c0 + u < n_runs;
      const float* pc = base + (size_t)(ok ? c0 + u : 0) * rstride;
      mc[u] = ok ? __ldcg(pc + D) : -INFINITY, lc[u] = ok ? __ldcg(pc + D + 1) : 0.f;
      oa[u] = ok ? __ldcg(reinterpret_cast<const float2*>(pc + tid * 4)) : make_float2(0.f, 0.f);
      ob[u] = ok ? __ldcg(reinterpret_cast<const float2*>(pc + tid * 4 + 2)) : make_float2(0.f, 0.f);
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const float wgt = (mc[u] == -INFINITY) ? 0.f : expf(mc[u] - m);
      l = fmaf(lc[u], wgt, l);
      acc[0] = fmaf(oa[u].x, wgt, acc[0]), acc[1] = fmaf(oa[u].y, wgt, acc[1]);
      acc[2] = fmaf(ob[u].x, wgt, acc[2]), acc[3] = fmaf(ob[u].y, wgt, acc[3]);
    }
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) store_split(p.aplanes + (size_t)row * 3 * HQ, HQ, h * D + tid * 4 + i, acc[i] / l);
}

}  // namespace ls
