// Inline-PTX building blocks of the tcgen05 first-level passes (sm_103a):
// mbarriers with bounded waits, TMA tile loads, shared-memory and instruction
// descriptors of kind::f16 MMAs, TMEM loads, and the host helpers the pass
// launchers share.
#pragma once

#include <cuda.h>

#include "plan.cuh"

namespace ttnn {
namespace tc {

constexpr int kTileM = 128;           // rows of M per tile (MMA M for D1)
constexpr int kTileN = 128;           // columns of M per tile (MMA M for D2)
constexpr int kMaxTiles = 16;         // column tiles per chunk (TMEM bounds it first)
constexpr int kSmemBudget = 232448 - 2048;   // 227 KB opt-in minus static shared memory
constexpr uint64_t kTimeoutNs = 2000000000ull;   // 2 s per wait

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ uint64_t gtimer() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}\n"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
// Bounded wait: false after limit_ns or when another role has aborted.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort,
                                          uint64_t limit_ns = kTimeoutNs) {
  if (mbar_try(bar, parity)) return true;
  const uint64_t t0 = gtimer();
  while (true) {
    if (mbar_try(bar, parity)) return true;
    if (*abort) return false;
    if (gtimer() - t0 > limit_ns) return false;
  }
}
// Bounded wait that ignores the abort flag (used to drain own work).
__device__ __forceinline__ bool mbar_drain(uint32_t bar, uint32_t parity) {
  const uint64_t t0 = gtimer();
  while (!mbar_try(bar, parity))
    if (gtimer() - t0 > kTimeoutNs) return false;
  return true;
}

__device__ __forceinline__ void tma_2d(uint32_t dst, const CUtensorMap* map, int x, int y,
                                       uint32_t bar, uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.L2::cache_hint"
      " [%0], [%1, {%2, %3}], [%4], %5;" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(bar), "l"(policy)
      : "memory");
}

// tcgen05 shared-memory descriptor: start, leading / stride byte offsets,
// fixed version bits 46-48 = 0b001, 128-byte swizzle (mode 2, bits 61-63).
__device__ __forceinline__ uint64_t sdesc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
  uint64_t d = (uint64_t)((saddr & 0x3FFFFu) >> 4);
  d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
  d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)2 << 61;
  return d;
}

// The descriptor of the same layout `bytes` (a multiple of 16) further on: one
// add to its low word.  (Shared memory ends below the address field's 256 KB,
// so nothing carries out of it.)  The thread that issues the MMAs builds two
// descriptors per MMA; made from the address each, that alone took longer
// than the MMA.
__device__ __forceinline__ uint64_t sdesc_at(uint64_t d, uint32_t bytes) {
  uint64_t r;
  asm("{\n\t.reg .b32 lo, hi;\n\tmov.b64 {lo, hi}, %1;\n\tadd.u32 lo, lo, %2;\n\t"
      "mov.b64 %0, {lo, hi};\n\t}\n"
      : "=l"(r)
      : "l"(d), "r"(bytes >> 4));
  return r;
}

// Instruction descriptor of kind::f16: D f32, A/B bf16, A K- or MN-major,
// B K-major, shape M x N.
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N, bool a_mn_major) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((a_mn_major ? 1u : 0u) << 15) |
         ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// The same for binary16 operands (formats 0).
__host__ __device__ constexpr uint32_t idesc_f16(int M, int N, bool a_mn_major) {
  return idesc_bf16(M, N, a_mn_major) & ~((1u << 7) | (1u << 10));
}

__device__ __forceinline__ void mma_bf16(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc,
                                         uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(d_tmem),
      "l"(a), "l"(b), "r"(idesc), "r"(accumulate));
}
__device__ __forceinline__ void mma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
               : "memory");
}
__device__ __forceinline__ void fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, "
      "%12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
}
__device__ __forceinline__ void tmem_wait_ld() {
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// Host helpers (pass_tc.cu).
// Raises a kernel's dynamic shared memory limit (to kSmemBudget unless its
// static shared memory leaves less), once per
// device.  Setting it per launch to the launch's own size would race between
// host threads launching the same kernel with different sizes.
ttnn_status smem_limit_once(const void* func, int slot, int bytes = kSmemBudget);
ttnn_status encode_map(CUtensorMap* m, const void* ptr, CUtensorMapDataType dt, int esize,
                       int64_t inner, int64_t outer, uint32_t box_inner, uint32_t box_outer,
                       CUtensorMapSwizzle sw);
int sm_count();
// SMs a first-level pass spreads its persistent CTAs over: all of them, or,
// with TTNN_FLAG_RESERVE_SMS, all but max(8, sketched nodes) (at most a
// quarter), which stay free for a recovery running on another stream.
int pass_sms(const ttnn_plan_s& P);
// D[i][w] = sum_k P[k][i][w] for w < wpad (rows i < rows).
ttnn_status launch_reduce_partials(const float* P, int K, int64_t stride_k, int64_t rows, int wpad,
                                   float* D, cudaStream_t st);

// D1 of a pass split into C column chunks: every chunk CTA writes its partial
// of a row block, each epilogue warp its 32 rows (row0 on) column by column:
// D1p = [C][nb * 4][wRpad][32], so a store is one whole line of 32 rows.
// (Row by row, as D1 is laid out, a warp's store touched 32 lines, and the
// load/store pipe they share with the converter warps cost a 48^5 binary32
// pass up to 32 of 245 us.)
__device__ __forceinline__ float* d1_partial(float* D1p, int64_t nb, int wRpad, int c, int64_t row0) {
  return D1p + ((int64_t)c * nb * kTileM + row0) * wRpad;
}
// Then it counts its arrival in *slot.  The warp that arrives last sums the C
// partials in chunk order (whoever is last) into D1, a lane 4 rows by 4 columns
// at a time, the loads of B partials in flight together, and drops the dead
// partial lines from L2 (`discard`: D1p is 128-byte aligned).  Called by all 32
// lanes after their own stores; no thread waits on another.
template <int B>
__device__ __forceinline__ void fold_d1_rows(int* slot, int C, const float* D1p, float* D1,
                                             int64_t nb, int wRpad, int64_t row0, int64_t nL,
                                             int discard, int lane) {
  __threadfence();
  __syncwarp();
  int last = 0;
  if (lane == 0) last = atomicAdd(slot, 1) == C - 1;
  last = __shfl_sync(0xffffffffu, last, 0);
  if (!last) return;
  __threadfence();
  const int i = lane & 7, j = lane >> 3;           // rows 4 i on, columns 4 j on (of 16)
  const int64_t cs = nb * kTileM * wRpad;          // chunk stride
  const float* src = D1p + row0 * wRpad;
  for (int cg = 0; cg < wRpad; cg += 16) {
    const float4* s4 = reinterpret_cast<const float4*>(src + (cg + 4 * j) * 32 + 4 * i);
    float4 acc[4];   // column 4 j + m: rows 4 i .. 4 i + 3
#pragma unroll
    for (int m = 0; m < 4; ++m) acc[m] = __ldcg(s4 + m * 8);
    for (int c0 = 1; c0 < C; c0 += B) {
      float4 v[B][4];
#pragma unroll
      for (int b = 0; b < B; ++b)
#pragma unroll
        for (int m = 0; m < 4; ++m)
          if (c0 + b < C) v[b][m] = __ldcg(s4 + (c0 + b) * (cs / 4) + m * 8);
#pragma unroll
      for (int b = 0; b < B; ++b) {
        if (c0 + b >= C) break;
#pragma unroll
        for (int m = 0; m < 4; ++m) {
          acc[m].x += v[b][m].x;
          acc[m].y += v[b][m].y;
          acc[m].z += v[b][m].z;
          acc[m].w += v[b][m].w;
        }
      }
    }
    const int64_t row = row0 + 4 * i;
    float* out = D1 + row * wRpad + cg + 4 * j;
    if (row < nL) *reinterpret_cast<float4*>(out) = make_float4(acc[0].x, acc[1].x, acc[2].x, acc[3].x);
    if (row + 1 < nL)
      *reinterpret_cast<float4*>(out + wRpad) = make_float4(acc[0].y, acc[1].y, acc[2].y, acc[3].y);
    if (row + 2 < nL)
      *reinterpret_cast<float4*>(out + 2 * wRpad) = make_float4(acc[0].z, acc[1].z, acc[2].z, acc[3].z);
    if (row + 3 < nL)
      *reinterpret_cast<float4*>(out + 3 * wRpad) = make_float4(acc[0].w, acc[1].w, acc[2].w, acc[3].w);
  }
  if (discard) {
    __syncwarp();
    for (int cc = 0; cc < C; ++cc)
      for (int l = lane; l < wRpad; l += 32)
        asm volatile("discard.global.L2 [%0], 128;" ::"l"((const char*)(src + cc * cs) + (int64_t)l * 128)
                     : "memory");
  }
}

}  // namespace tc
}  // namespace ttnn
