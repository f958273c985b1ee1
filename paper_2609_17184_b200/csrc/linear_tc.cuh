// Weight-streaming linear map on the fifth-generation tensor cores: y[m][n] = sum_k x[m][k] W[n][k].
//
// The same contraction as the skinny GEMMs of the decode pass (Sec. 4.2 step 1: the token-at-depth rows are the
// narrow side, the shared weights the wide side that streams from HBM), built from the Blackwell pieces: tiles of
// the row-major weights and of the activation planes arrive by TMA (cp.async.bulk.tensor, 128-byte swizzle) in a
// ring of shared-memory stages guarded by mbarriers; one thread issues tcgen05.mma (128 weight rows x up to 64 token
// columns, K = 16 per instruction) with the accumulator in tensor memory; four warps read it back with tcgen05.ld.
// Activations are fp32 split exactly into three bf16 planes; the planes are stacked as 3 MP columns of one MMA per
// k-step (three accumulator chains, as in the mma.sync kernels) and folded hi + (mid + lo) when the accumulator is read.
// K may be split over blockIdx.y; the partial sums are added in split order by a second kernel (no atomics).  Passes of
// more than 64 token columns put one group of 64 columns in each blockIdx.z plane.
//
// Used by the stand-alone operator loopspec_op_linear_tc, by the prefill passes and by the decode passes that carry 9 or
// more rows (tc_epilogue_kernel then applies the fused epilogue of the GEMM); decode passes of up to 8 rows run
// gemm_bf16_kernel, whose launch is cheaper than this pair's.
#pragma once
#include <cuda.h>

#include "common.cuh"

namespace ls {

constexpr int TC_THREADS = 128;
constexpr int TC_BM = 128;         // weight rows per CTA = rows of one MMA
constexpr int TC_BK = 64;          // k per stage: 64 bf16 = one 128-byte swizzled row
constexpr int TC_MAX_STAGES = 8;
constexpr int TC_SMEM_MAX = 101 * 1024;  // most dynamic shared memory any launch of linear_tc_kernel asks for
constexpr long long TC_WAIT_CYCLES = 400000000LL;  // ~0.2 s: a wait that runs this long gives up and raises the flag

struct LinearTcParams {
  float* out;          // [n_split][M][N] partial sums (n_split == 1: y itself)
  int M, MP, N, K;     // MP = M rounded up to 16: columns of the MMA
  int kb_per_split;    // 64-wide k-blocks per blockIdx.y
  int stages;
  int* err;            // flag the host reads: set to err_code when a bounded wait ran out
  int err_code;
  int x3d;             // 0: x planes stacked [3][MP][K], one box; 1: the decode pass's layout [column][3][x_ld], a
                       // three-dimensional map (k, plane, column) and one box per plane
  int row0;            // x3d: first column of the map this launch carries; blockIdx.z adds group_cols to it and
  int group_cols;      //      group_stride floats to `out` (passes wider than one MMA's columns: one grid plane per
  long long group_stride;  //  group of columns)
  const int* n_live;   // x3d: number of live columns of the pass (may be null); a group beyond it has nothing to do
  long long wait_cycles;
  int stop_kb;         // test hook: no CTA requests its k-blocks from this one on (INT_MAX: all are), so that the waits for them run out
};

__device__ __forceinline__ unsigned tc_smem_u32(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void tc_mbar_init(unsigned bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void tc_mbar_expect_tx(unsigned bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
// bounded wait on a phase parity: false when it gave up
__device__ __forceinline__ bool tc_mbar_wait(unsigned bar, unsigned parity, long long limit) {
  const long long t0 = clock64();
  for (;;) {
    unsigned ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    if (ok) return true;
    if (clock64() - t0 > limit) return false;
  }
}
__device__ __forceinline__ void tc_tma_load_2d(unsigned dst, const CUtensorMap* map, unsigned bar, int x, int y) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];" ::"r"(dst),
      "l"(reinterpret_cast<unsigned long long>(map)), "r"(bar), "r"(x), "r"(y)
      : "memory");
}
__device__ __forceinline__ void tc_tma_load_3d(unsigned dst, const CUtensorMap* map, unsigned bar, int x, int y, int z) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];" ::"r"(dst),
      "l"(reinterpret_cast<unsigned long long>(map)), "r"(bar), "r"(x), "r"(y), "r"(z)
      : "memory");
}
// shared-memory matrix descriptor: K-major tile of 128-byte rows, 128-byte swizzle, 8-row groups 1024 bytes apart
__device__ __forceinline__ unsigned long long tc_smem_desc(unsigned addr) {
  unsigned long long d = 0;
  d |= (unsigned long long)((addr >> 4) & 0x3FFF);
  d |= (unsigned long long)(1024 >> 4) << 32;  // stride between 8-row groups
  d |= 1ull << 46;                             // descriptor version of this architecture
  d |= 2ull << 61;                             // 128-byte swizzle
  return d;
}
// instruction descriptor: bf16 x bf16 -> fp32, both operands K-major, M x N
__host__ __device__ constexpr unsigned tc_idesc(int M, int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((unsigned)(N >> 3) << 17) | ((unsigned)(M >> 4) << 24);
}
__device__ __forceinline__ void tc_mma(unsigned d_tmem, unsigned long long adesc, unsigned long long bdesc, unsigned idesc,
                                       unsigned accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\ttcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// One lane of a converged warp, always the same.  tcgen05.mma takes its operands from uniform registers: issued under a branch on
// the lane number every MMA first moves them there, about 60 cycles each; under this one the compiler keeps them uniform.
__device__ __forceinline__ bool tc_elect_one() {
  unsigned e;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(e));
  return e != 0;
}
__device__ __forceinline__ void tc_commit(unsigned bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

__host__ __device__ constexpr int tc_stage_bytes(int MP) { return TC_BM * TC_BK * 2 + 3 * MP * TC_BK * 2; }
// Dynamic shared memory of a launch: the ring, and for more than 128 accumulator columns (256 of tensor memory) enough that no third CTA
// fits an SM: it would hold its slot in the tensor-memory allocation until another CTA ends, ahead of the kernels that could run there
// [decode passes of 35 to 48 rows, 2 stages of 34 KB each: 5 sequences of 260 positions 1.89 -> 1.56 ms per pass, one live 1.61 -> 1.41].
// (Fewer columns: four and more CTAs share the 512 columns, and the rings keep them below that.)
inline size_t tc_smem_bytes(int MP, int stages) {
  const size_t ring = (size_t)stages * tc_stage_bytes(MP) + 1024;
  return 3 * MP > 128 && ring < 78 * 1024 ? 78 * 1024 : ring;
}

__global__ void __launch_bounds__(TC_THREADS) linear_tc_kernel(const __grid_constant__ CUtensorMap map_w,
                                                               const __grid_constant__ CUtensorMap map_x,
                                                               const __grid_constant__ LinearTcParams p) {
  extern __shared__ unsigned char tc_smem_raw[];
  __shared__ __align__(8) unsigned long long s_full[TC_MAX_STAGES], s_empty[TC_MAX_STAGES], s_done;
  __shared__ unsigned s_tmem;
  __shared__ int s_fail;

  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;  // (warp: uniform to the compiler)
  const unsigned base = (tc_smem_u32(tc_smem_raw) + 1023u) & ~1023u;  // swizzled tiles sit on 1024-byte boundaries
  const int stage_bytes = tc_stage_bytes(p.MP);
  const int n0 = blockIdx.x * TC_BM;
  const int kb0 = blockIdx.y * p.kb_per_split;
  const int n_kb = min(p.kb_per_split, p.K / TC_BK - kb0);
  // the three planes of the activations are three groups of MP accumulator columns: one MMA of N = 3 MP per k-step
  // (three separate chains, as in the mma.sync kernels), folded hi + (mid + lo) when the accumulator is read
  const unsigned tmem_cols = 3 * p.MP <= 64 ? 64u : (3 * p.MP <= 128 ? 128u : 256u);

  if (tid == 32) {  // the producer fetches the two tensor maps while the barriers are set up
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<unsigned long long>(&map_w)) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<unsigned long long>(&map_x)) : "memory");
  }
  if (tid == 0) {
    for (int s = 0; s < p.stages; ++s) tc_mbar_init(tc_smem_u32(&s_full[s]), 1), tc_mbar_init(tc_smem_u32(&s_empty[s]), 1);
    tc_mbar_init(tc_smem_u32(&s_done), 1);
    s_fail = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  __syncthreads();
  pdl_launch_dependents();
  const int row0 = p.row0 + (int)blockIdx.z * p.group_cols;
  // columns that carry a token (final before the pass starts; uniform over the CTA): the others are neither loaded for nor written.  A pass
  // whose group is empty - the second group of a small batch, the prelude and coda blocks of a Raven pass without rows at their
  // depths - requests no weights at all
  const int live = p.n_live ? min(p.M, *p.n_live - row0) : p.M;
  if (live <= 0) {
    pdl_wait();  // a kernel that ended before its predecessor would release its own dependents too early
    return;
  }
  // The weights are constants, so the first ring-full of weight tiles is requested ahead of the predecessor's
  // completion - and while warp 0 still allocates the tensor memory; the activation tiles (which the predecessor may
  // still be writing) follow after the dependency wait, on the same barriers.
  const int n_load = min(n_kb, p.stop_kb), pre = min(p.stages, n_load);
  if (tid == 32) {
    for (int kb = 0; kb < pre; ++kb) {
      const unsigned bar = tc_smem_u32(&s_full[kb]);
      tc_mbar_expect_tx(bar, (unsigned)stage_bytes);
      tc_tma_load_2d(base + kb * stage_bytes, &map_w, bar, (kb0 + kb) * TC_BK, n0);
    }
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tc_smem_u32(&s_tmem)), "r"(tmem_cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const unsigned tmem = s_tmem;

  pdl_wait();
  auto load_x = [&](unsigned b, unsigned bar, int k) {  // the three planes of the activations, plane pl at b + pl * MP * 128
    if (p.x3d) {
#pragma unroll
      for (int pl = 0; pl < 3; ++pl) tc_tma_load_3d(b + pl * p.MP * TC_BK * 2, &map_x, bar, k, pl, row0);
    } else {
      tc_tma_load_2d(b, &map_x, bar, k, 0);
    }
  };
  if (tid == 32 && n_kb > 0) {
    // ---- producer: one thread keeps the ring of stages filled by TMA ----
    for (int kb = 0; kb < pre; ++kb)
      load_x(base + kb * stage_bytes + TC_BM * TC_BK * 2, tc_smem_u32(&s_full[kb]), (kb0 + kb) * TC_BK);
    bool ok = true;
    for (int kb = pre; kb < n_load && ok; ++kb) {
      const int s = kb % p.stages;
      ok = tc_mbar_wait(tc_smem_u32(&s_empty[s]), ((kb / p.stages) - 1) & 1, p.wait_cycles);  // the stage's MMAs are done
      if (!ok) break;
      const unsigned bar = tc_smem_u32(&s_full[s]);
      const unsigned a = base + s * stage_bytes, b = a + TC_BM * TC_BK * 2;
      tc_mbar_expect_tx(bar, (unsigned)stage_bytes);
      tc_tma_load_2d(a, &map_w, bar, (kb0 + kb) * TC_BK, n0);
      load_x(b, bar, (kb0 + kb) * TC_BK);
    }
    if (!ok) s_fail = 1, *p.err = p.err_code;
  }
  __syncwarp();  // (the other lanes do not poll for the end next to the producer)
  if (warp == 0 && n_kb > 0) {
    // ---- MMA issuer: one elected lane, the accumulator lives in tensor memory ----
    const unsigned idesc = tc_idesc(TC_BM, 3 * p.MP);
    // No lane leaves the loop when a wait runs out - the others would wait for it, without a bound, at the next instruction of the
    // whole warp: the rest of the k-blocks is walked without MMAs, and every barrier still receives its arrival.
    bool ok = true;
    for (int kb = 0; kb < n_kb; ++kb) {
      const int s = kb % p.stages;
      if (!tc_mbar_wait(tc_smem_u32(&s_full[s]), (kb / p.stages) & 1, ok ? p.wait_cycles : 0)) ok = false;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      if (tc_elect_one()) {
        const unsigned a = base + s * stage_bytes, b = a + TC_BM * TC_BK * 2;
        const unsigned long long adesc = tc_smem_desc(a);
        const unsigned long long bdesc = tc_smem_desc(b);  // rows pl * MP + column: the hi, mid, lo planes stacked
        if (ok) {
#pragma unroll
          for (int ks = 0; ks < TC_BK / 16; ++ks) tc_mma(tmem, adesc + 2 * ks, bdesc + 2 * ks, idesc, (kb | ks) != 0);
        }
        tc_commit(tc_smem_u32(&s_empty[s]));  // arrives when the MMAs issued so far have read their operands
        if (kb == n_kb - 1) {
          if (!ok) s_fail = 1, *p.err = p.err_code, __threadfence_block();
          tc_commit(tc_smem_u32(&s_done));
        }
      }
      __syncwarp();
    }
  }
  // everyone: the accumulator is complete when the last commit arrives.  It is read either way (the loads are the whole warp's); a
  // lane that does not have it complete stores nothing.
  const bool have = n_kb > 0 && tc_mbar_wait(tc_smem_u32(&s_done), 0, p.wait_cycles) && *const_cast<volatile int*>(&s_fail) == 0;
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const int n = n0 + warp * 32 + lane;  // this thread's weight row = its TMEM lane
  float* out = p.out + (size_t)blockIdx.z * p.group_stride + (size_t)blockIdx.y * p.M * p.N;
  if (n_kb <= 0) {
    for (int m = 0; m < live; ++m)
      if (n < p.N) out[(size_t)m * p.N + n] = 0.f;
  } else {
    for (int c0 = 0; c0 < live; c0 += 16) {
      unsigned w[3][16];
#pragma unroll
      for (int pl = 0; pl < 3; ++pl) {
        const unsigned taddr = tmem + ((unsigned)(warp * 32) << 16) + (unsigned)(pl * p.MP + c0);
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
            : "=r"(w[pl][0]), "=r"(w[pl][1]), "=r"(w[pl][2]), "=r"(w[pl][3]), "=r"(w[pl][4]), "=r"(w[pl][5]), "=r"(w[pl][6]),
              "=r"(w[pl][7]), "=r"(w[pl][8]), "=r"(w[pl][9]), "=r"(w[pl][10]), "=r"(w[pl][11]), "=r"(w[pl][12]),
              "=r"(w[pl][13]), "=r"(w[pl][14]), "=r"(w[pl][15])
            : "r"(taddr)
            : "memory");
      }
      asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
      unsigned v[16];
#pragma unroll
      for (int j = 0; j < 16; ++j)
        v[j] = __float_as_uint(__uint_as_float(w[0][j]) + (__uint_as_float(w[1][j]) + __uint_as_float(w[2][j])));
#pragma unroll
      for (int j = 0; j < 16; ++j)
        if (c0 + j < live && n < p.N && have) out[(size_t)(c0 + j) * p.N + n] = __uint_as_float(v[j]);
    }
    if (!have) s_fail = 1, *p.err = p.err_code;
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0) {
    // a wait that gave up may have left copies in flight: give them a bounded time to land before the memory is freed
    if (s_fail) {
      const long long t0 = clock64();
      while (clock64() - t0 < 2000000LL) {
      }
    }
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(tmem_cols) : "memory");
  }
}

// x fp32 [M][K] -> planes bf16 [3][MP][K] (rows M..MP-1 zero); clears the flag of the kernel that follows.  Eight values a
// thread (K is a multiple of 64), one CTA per row and 2048 of k.
inline int tc_split_blocks(int K) { return (K + 2047) / 2048; }
__global__ void __launch_bounds__(256) tc_split_kernel(const float* __restrict__ x, __nv_bfloat16* __restrict__ planes, int M, int MP, int K, int* err) {
  pdl_launch_dependents();
  const int m = blockIdx.x, k = (blockIdx.y * 256 + threadIdx.x) * 8;
  if (m == 0 && k == 0) *err = 0;
  if (k >= K) return;
  unsigned short s[3][8];
  float v[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  if (m < M) {
    const float* src = x + (size_t)m * K + k;
    if ((reinterpret_cast<unsigned long long>(x) & 15) == 0) {
      const float4 a = *reinterpret_cast<const float4*>(src), b = *reinterpret_cast<const float4*>(src + 4);
      v[0] = a.x, v[1] = a.y, v[2] = a.z, v[3] = a.w, v[4] = b.x, v[5] = b.y, v[6] = b.z, v[7] = b.w;
    } else {
      for (int i = 0; i < 8; ++i) v[i] = src[i];
    }
  }
#pragma unroll
  for (int i = 0; i < 8; ++i) split3(v[i], s[0][i], s[1][i], s[2][i]);
#pragma unroll
  for (int p = 0; p < 3; ++p)
    *reinterpret_cast<uint4*>(planes + ((size_t)p * MP + m) * K + k) =
        make_uint4(s[p][0] | ((unsigned)s[p][1] << 16), s[p][2] | ((unsigned)s[p][3] << 16), s[p][4] | ((unsigned)s[p][5] << 16), s[p][6] | ((unsigned)s[p][7] << 16));
}

// y = sum over the k-splits, in split order (MN is a multiple of 8: four values a thread and step where y is 16-byte aligned)
__global__ void __launch_bounds__(256) tc_sum_splits_kernel(const float* __restrict__ part, float* __restrict__ y, size_t MN, int n_split) {
  pdl_wait();
  const size_t step = (size_t)gridDim.x * blockDim.x * 4;
  for (size_t i = (blockIdx.x * (size_t)blockDim.x + threadIdx.x) * 4; i < MN; i += step) {
    float4 v = __ldcg(reinterpret_cast<const float4*>(part + i));
    for (int s = 1; s < n_split; ++s) {
      const float4 t = __ldcg(reinterpret_cast<const float4*>(part + (size_t)s * MN + i));
      v.x += t.x, v.y += t.y, v.z += t.z, v.w += t.w;
    }
    if ((reinterpret_cast<unsigned long long>(y) & 15) == 0) *reinterpret_cast<float4*>(y + i) = v;
    else y[i] = v.x, y[i + 1] = v.y, y[i + 2] = v.z, y[i + 3] = v.w;
  }
}

}  // namespace ls
