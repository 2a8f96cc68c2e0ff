// GEMM on the tcgen05 tensor cores with the large operand loaded by converter
// warps instead of TMA, for first-level products of tensors whose rows TMA
// cannot address (a stride that is not a multiple of 16 bytes) and of
// binary32 boxes.  The SIMT GEMM these took before ran at 12.5 TFLOP/s of the
// 80 the FMA pipes have; here the tensor is read at HBM speed and the
// products run on the tensor cores.
//
// Precision.  bfloat16 operands are multiplied as they are.  A binary32
// operand is cut into three bfloat16 pieces that sum to it exactly (8 + 8 + 8
// significand bits, each cut towards zero, so no piece overflows); the six
// products down to 2^-16 of the leading one are formed, the other three
// (2^-24 and below) are left out.  The tensor core truncates when it adds to
// its binary32 accumulator, so chains are short: the leading products of 128
// k go into one accumulator, those of each lower order into another, and the
// epilogue warps add them to registers with rounding to nearest.  The pieces
// of B sit below one another in shared memory, so piece i of A meets all the
// pieces of B it is multiplied with in one MMA of up to three times the
// columns: the MMAs are bound by reading their operands from shared memory
// (about 100 cycles for 128 x 64 x 16), and A is read three times per k step
// instead of six.
//
// Warp roles: warp 0 copies B tiles by TMA, warp 1 owns TMEM and issues the
// MMAs, warps 2-5 drain accumulators (TMEM lane quarter = warp % 4), the
// other 16 (8) load, convert and store A tiles (128-byte swizzle).  Every
// wait is bounded; on expiry the kernel sets an error bit, drains its own
// copies and MMAs, frees TMEM and returns.
#include <cuda_bf16.h>

#include <algorithm>

#include "gemm_tc.cuh"
#include "tc_ptx.cuh"

namespace ttnn {
namespace tc {

constexpr int kTcgMaxN = 80;      // columns an epilogue thread accumulates
// Converter warps: 16 hide the most latency; products wider than 64 columns
// need the registers of eight of them for the epilogue's sums.
template <int NW>
__host__ __device__ constexpr int tcg_conv_warps() { return NW <= 64 ? 16 : 8; }
template <int NW>
__host__ __device__ constexpr int tcg_threads() { return 192 + 32 * tcg_conv_warps<NW>(); }
constexpr int kTcgMaxStages = 6;

struct TcgParams {
  const void* A;
  int64_t lda, I, K;
  int nI, nkt;           // row tiles, k tiles
  int Npad, stages;
  int group;             // k tiles per drain of the accumulators
  float* C;              // [I][Npad]
  float* part;           // pieces [2 grid][128][Npad]
  int* err;
  uint64_t wait_ns;
};

// Shape of a form: pieces per element, k of a tile, accumulators, converter
// groups (each converts a tile in turn; at most the number of stages, so that
// a group never waits two phases ahead of a barrier).
template <typename T>
struct Form;
template <>
struct Form<uint16_t> {
  static constexpr int NS = 1, KT = 128, NACC = 1, NG = 1;
};
template <>
struct Form<float> {
  static constexpr int NS = 3, KT = 64, NACC = 3, NG = 2;
};

// Two adjacent elements of a row, as loaded.  VEC: extents, stride and base
// are even, so a pair is one aligned load and never straddles an edge.
template <typename T, bool VEC>
struct Pair;
template <>
struct Pair<uint16_t, true> {
  uint32_t v;
  __device__ void load(const uint16_t* p, bool a, bool) {
    v = a ? __ldg(reinterpret_cast<const uint32_t*>(p)) : 0u;
  }
  __device__ uint32_t word() const { return v; }
};
template <>
struct Pair<uint16_t, false> {
  uint16_t x, y;
  __device__ void load(const uint16_t* p, bool a, bool b) {
    x = a ? __ldg(p) : (uint16_t)0;
    y = b ? __ldg(p + 1) : (uint16_t)0;
  }
  __device__ uint32_t word() const { return (uint32_t)x | ((uint32_t)y << 16); }
};
template <bool VEC>
struct Pair<float, VEC> {
  float x, y;
  __device__ void load(const float* p, bool a, bool b) {
    if (VEC) {
      const float2 v = a ? __ldg(reinterpret_cast<const float2*>(p)) : make_float2(0.f, 0.f);
      x = v.x;
      y = v.y;
    } else {
      x = a ? __ldg(p) : 0.f;
      y = b ? __ldg(p + 1) : 0.f;
    }
  }
};

// The three pieces of two binary32 values, packed (x in the low half).  The
// rest of an infinity is NaN: a non-finite entry makes every result it
// reaches NaN.
__device__ __forceinline__ void cut3(float x, float y, uint32_t* w) {
  const uint32_t ux = __float_as_uint(x), uy = __float_as_uint(y);
  w[0] = __byte_perm(ux, uy, 0x7632);
  x -= __uint_as_float(ux & 0xFFFF0000u);
  y -= __uint_as_float(uy & 0xFFFF0000u);
  const uint32_t vx = __float_as_uint(x), vy = __float_as_uint(y);
  w[1] = __byte_perm(vx, vy, 0x7632);
  x -= __uint_as_float(vx & 0xFFFF0000u);
  y -= __uint_as_float(vy & 0xFFFF0000u);
  w[2] = __byte_perm(__float_as_uint(x), __float_as_uint(y), 0x7632);
}

__device__ __forceinline__ void st_shared(uint32_t addr, uint32_t v) {
  asm volatile("st.shared.b32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7])
      : "r"(taddr));
}

// NW: the columns an epilogue thread holds sums of (Npad <= NW).
template <typename T, bool MN, bool VEC, int NW>
__global__ void __launch_bounds__(tcg_threads<NW>(), 1)
    tcg_kernel(const __grid_constant__ CUtensorMap mapB, const TcgParams p) {
  using F = Form<T>;
  constexpr int NS = F::NS, KT = F::KT, NACC = F::NACC;
  constexpr int R = MN ? KT : kTileM;            // tile rows in memory order
  constexpr int CB = MN ? 2 : KT / 64;           // 64-column boxes of a row
  constexpr int NG = F::NG;                      // converter groups, a tile each in turn
  constexpr int NCW = tcg_conv_warps<NW>() / NG; // warps of a group
  constexpr int RW = R / NCW;                    // rows of a converter warp (4, 8 or 16)
  constexpr int NP = RW * CB;                    // pairs of a converter thread per tile
  constexpr uint32_t kBox = R * 128;             // bytes of a box
  constexpr uint32_t kPiece = kBox * CB;         // bytes of one piece of the tile
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t bar_a[kTcgMaxStages], bar_b[kTcgMaxStages], bar_empty[kTcgMaxStages];
  __shared__ __align__(8) uint64_t bar_full[2], bar_free[2], bar_done;
  __shared__ uint32_t tmem_slot;
  __shared__ volatile int abort_flag;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  const uint32_t base = smem_u32(smem);
  const int S = p.stages;
  const uint32_t b_piece = (uint32_t)p.Npad * KT * 2;
  const uint32_t stage_bytes = NS * (kPiece + b_piece);
  // The (row tile, k tile) grid in row-major order is cut into gridDim.x even
  // ranges, one per CTA.  Row tiles within one range go to C; only the first
  // and the last of a range can be pieces of a tile (slots 2 c and 2 c + 1 of
  // CTA c), which are summed afterwards in CTA order.
  const int64_t total = (int64_t)p.nI * p.nkt;
  const int64_t u0 = total * blockIdx.x / gridDim.x, u1 = total * (blockIdx.x + 1) / gridDim.x;
  const int i0 = (int)(u0 / p.nkt), i1 = u1 > u0 ? (int)((u1 - 1) / p.nkt) + 1 : i0;

  if (threadIdx.x == 0) {
    abort_flag = 0;
    for (int s = 0; s < S; ++s) {
      mbar_init(smem_u32(&bar_a[s]), NCW);
      mbar_init(smem_u32(&bar_b[s]), 1);
      mbar_init(smem_u32(&bar_empty[s]), 1);
    }
    for (int k = 0; k < 2; ++k) {
      mbar_init(smem_u32(&bar_full[k]), 1);
      mbar_init(smem_u32(&bar_free[k]), 4);
    }
    mbar_init(smem_u32(&bar_done), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(&tmem_slot)),
                 "r"(512u));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = tmem_slot;

  // this CTA's k tiles of row tile `it`
  auto range = [&](int it, int* kt0, int* kt1) {
    const int64_t r = (int64_t)it * p.nkt;
    *kt0 = (int)(max(u0, r) - r);
    *kt1 = (int)(min(u1, r + p.nkt) - r);
  };

  if (warp == 0) {
    if (lane == 0) {
      // ---------------- B tiles by TMA ----------------
      uint64_t pol_keep;
      asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(pol_keep));
      int stage = 0;
      uint32_t ph = 0, used = 0, last_ph = 0;
      bool ok = true;
      for (int it = i0; it < i1 && ok; ++it) {
        int kt0, kt1;
        range(it, &kt0, &kt1);
        for (int kt = kt0; kt < kt1; ++kt) {
          ok = mbar_wait(smem_u32(&bar_empty[stage]), ph ^ 1, &abort_flag, p.wait_ns);
          if (!ok) break;
          const uint32_t bar = smem_u32(&bar_b[stage]);
          const uint32_t sb = base + stage * stage_bytes + NS * kPiece;
          mbar_expect_tx(bar, NS * b_piece);
#pragma unroll
          for (int s = 0; s < NS; ++s)
#pragma unroll
            for (int h = 0; h < KT / 64; ++h)
              tma_2d(sb + s * b_piece + h * (b_piece / (KT / 64)), &mapB, kt * KT + h * 64,
                     s * p.Npad, bar, pol_keep);
          used |= 1u << stage;
          last_ph = (last_ph & ~(1u << stage)) | (ph << stage);
          if (++stage == S) {
            stage = 0;
            ph ^= 1;
          }
        }
      }
      if (!ok) {
        abort_flag = 1;
        atomicOr(p.err, 1);
      }
      for (int s = 0; s < S; ++s)
        if (((used >> s) & 1u) && !mbar_drain(smem_u32(&bar_b[s]), (last_ph >> s) & 1u))
          atomicOr(p.err, 2);
    }
  } else if (warp == 1) {
    if (lane == 0) {
      // ---------------- MMA issuer ----------------
      static_assert(NS == 1 || KT == 64, "the pieces of a B tile are adjacent rows of one box");
      int stage = 0, buf = 0;
      uint32_t ph = 0, fph = 1;
      bool ok = true;
      for (int it = i0; it < i1 && ok; ++it) {
        int kt0, kt1;
        range(it, &kt0, &kt1);
        for (int g0 = kt0; g0 < kt1 && ok; g0 += p.group) {
          ok = mbar_wait(smem_u32(&bar_free[buf]), fph, &abort_flag, p.wait_ns);
          if (!ok) break;
          fence_after();
          const uint32_t d = tmem + buf * NACC * p.Npad;
          const int g1 = min(g0 + p.group, kt1);
          for (int kt = g0; kt < g1; ++kt) {
            ok = mbar_wait(smem_u32(&bar_a[stage]), ph, &abort_flag, p.wait_ns) &&
                 mbar_wait(smem_u32(&bar_b[stage]), ph, &abort_flag, p.wait_ns);
            if (!ok) break;
            fence_after();
            const uint32_t sa = base + stage * stage_bytes;
            const uint32_t sb = sa + NS * kPiece;
#pragma unroll
            for (int ia = 0; ia < NS; ++ia) {
              // piece ia of A against pieces 0 .. NS - 1 - ia of B: orders ia .. NS - 1
              const uint32_t id = idesc_bf16(kTileM, (NS - ia) * p.Npad, MN);
#pragma unroll
              for (int kk = 0; kk < KT / 16; ++kk) {
                const uint64_t da =
                    MN ? sdesc(sa + ia * kPiece + kk * 2048, kBox, 1024)
                       : sdesc(sa + ia * kPiece + (kk >> 2) * kBox + (kk & 3) * 32, 16, 1024);
                const uint64_t db =
                    sdesc(sb + (kk >> 2) * (p.Npad * 128) + (kk & 3) * 32, 16, 1024);
                mma_bf16(d + ia * p.Npad, da, db, id, kt > g0 || kk > 0 || ia > 0);
              }
            }
            mma_commit(smem_u32(&bar_empty[stage]));
            if (++stage == S) {
              stage = 0;
              ph ^= 1;
            }
          }
          if (!ok) break;
          mma_commit(smem_u32(&bar_full[buf]));
          buf ^= 1;
          if (buf == 0) fph ^= 1;
        }
      }
      if (!ok) {
        abort_flag = 1;
        atomicOr(p.err, 4);
      }
      mma_commit(smem_u32(&bar_done));
    }
  } else if (warp >= 6) {
    // ---------------- converters ----------------
    const int cw = (warp - 6) % NCW, grp = (warp - 6) / NCW;
    const T* A = (const T*)p.A;
    const int64_t rows = MN ? p.K : p.I, cols = MN ? p.I : p.K;
    int stage = 0;
    uint32_t ph = 0;
    bool ok = true;
    // v holds a tile's pairs; each is reloaded for the next tile as soon as
    // it is stored, so a whole tile of loads is in flight per warp
    Pair<T, VEC> v[NP];
    int it = i0, kt = 0, kt1 = 0;
    const T* src = nullptr;
    int nrow = 0, ncol = 0;     // valid rows of the warp, valid columns from the lane's on
    auto aim = [&]() {
      const int64_t r0 = (MN ? kt * (int64_t)KT : it * (int64_t)kTileM) + cw * RW;
      const int64_t c0 = (MN ? it * (int64_t)kTileM : kt * (int64_t)KT) + 2 * lane;
      src = A + r0 * p.lda + c0;
      nrow = (int)max((int64_t)0, min((int64_t)RW, rows - r0));
      ncol = (int)max((int64_t)0, min((int64_t)256, cols - c0));
    };
    // every pair of the warp inside the operand: no bounds on the loads
    auto interior = [&]() {
      return __all_sync(0xffffffffu, nrow == RW && ncol > (CB - 1) * 64 + 1);
    };
    auto load = [&](int q, bool all) {
      const int rr = q / CB, c = (q % CB) * 64;
      v[q].load(src + (int64_t)rr * p.lda + c, all || (rr < nrow && c < ncol),
                all || (rr < nrow && c + 1 < ncol));
    };
    // on by n tiles of this CTA's range
    auto advance = [&](int n) {
      kt += n;
      while (it < i1 && kt >= kt1) {
        n = kt - kt1;
        if (++it < i1) {
          range(it, &kt, &kt1);
          kt += n;
        }
      }
    };
    if (it < i1) {
      range(it, &kt, &kt1);
      advance(grp);
      stage = grp % S;
      ph = (uint32_t)(grp / S) & 1u;
    }
    if (it < i1) {
      aim();
#pragma unroll
      for (int q = 0; q < NP; ++q) load(q, false);
    }
    // the 16-byte chunk c of row y sits at chunk c ^ (y & 7) of its 128-byte row
    const uint32_t at = (uint32_t)(cw * RW * 128 + 4 * lane);
    while (it < i1) {
      advance(NG);
      if (it < i1) aim();
      else nrow = 0;
      const bool all = interior();
      ok = mbar_wait(smem_u32(&bar_empty[stage]), ph ^ 1, &abort_flag, p.wait_ns);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      const uint32_t dst = base + stage * stage_bytes + at;
      auto store = [&](int q) {
        const int rr = q / CB;
        const uint32_t sw = ((uint32_t)((RW == 4 ? (cw & 1) * 4 : 0) + rr) & 7u) << 4;
        const uint32_t o = (dst ^ sw) + (q % CB) * kBox + rr * 128;
        if constexpr (NS == 1) {
          st_shared(o, v[q].word());
        } else {
          uint32_t w[3];
          cut3(v[q].x, v[q].y, w);
#pragma unroll
          for (int s = 0; s < 3; ++s) st_shared(o + s * kPiece, w[s]);
        }
      };
      if (all) {
#pragma unroll
        for (int q = 0; q < NP; ++q) {
          store(q);
          load(q, true);
        }
      } else {
#pragma unroll
        for (int q = 0; q < NP; ++q) {
          store(q);
          load(q, false);
        }
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&bar_a[stage]));
      for (int k = 0; k < NG; ++k)
        if (++stage == S) {
          stage = 0;
          ph ^= 1;
        }
    }
    if (!ok) {
      abort_flag = 1;
      atomicOr(p.err, 64);
    }
  } else {
    // ---------------- epilogue (warps 2..5) ----------------
    const int q = warp & 3;
    const uint32_t lane_off = (uint32_t)(32 * q) << 16;
    int buf = 0;
    uint32_t fph = 0;
    bool ok = true;
    for (int it = i0; it < i1 && ok; ++it) {
      int kt0, kt1;
      range(it, &kt0, &kt1);
      float acc[NW];
#pragma unroll
      for (int c = 0; c < NW; ++c) acc[c] = 0.f;
      for (int g0 = kt0; g0 < kt1; g0 += p.group) {
        ok = mbar_wait(smem_u32(&bar_full[buf]), fph, &abort_flag, p.wait_ns);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        fence_after();
        const uint32_t d = tmem + lane_off + buf * NACC * p.Npad;
#pragma unroll
        for (int cg = 0; cg < NW; cg += 8) {
          if (cg >= p.Npad) continue;
          uint32_t x[NACC][8];
#pragma unroll
          for (int o = 0; o < NACC; ++o) tmem_ld8(d + o * p.Npad + cg, x[o]);
          tmem_wait_ld();
#pragma unroll
          for (int c = 0; c < 8; ++c) {
            float v = __uint_as_float(x[NACC - 1][c]);
#pragma unroll
            for (int o = NACC - 2; o >= 0; --o) v += __uint_as_float(x[o][c]);
            acc[cg + c] += v;
          }
        }
        fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&bar_free[buf]));
        buf ^= 1;
        if (buf == 0) fph ^= 1;
      }
      if (!ok) break;
      const bool whole = kt0 == 0 && kt1 == p.nkt;
      const int64_t row = (int64_t)it * kTileM + 32 * q + lane;
      if (row < p.I) {
        float* dst = whole ? p.C + row * p.Npad
                           : p.part + ((int64_t)(2 * blockIdx.x + (it > i0)) * kTileM + 32 * q + lane) * p.Npad;
        float4* out = reinterpret_cast<float4*>(dst);
#pragma unroll
        for (int c = 0; c < NW / 4; ++c)
          if (4 * c < p.Npad) out[c] = make_float4(acc[4 * c], acc[4 * c + 1], acc[4 * c + 2], acc[4 * c + 3]);
      }
    }
    if (!ok) {
      abort_flag = 1;
      atomicOr(p.err, 8);
    }
  }
  // all MMAs must be complete before TMEM is released
  if (warp == 1 && lane == 0) {
    if (!mbar_drain(smem_u32(&bar_done), 0)) atomicOr(p.err, 32);
  }
  fence_before();
  __syncthreads();
  fence_after();
  if (warp == 1)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u));
}

// The B operands as the kernel's TMA reads them: [NS][Npad][Kpad] bfloat16,
// zero beyond the operand.
struct PrepJob {
  const void* src;
  uint16_t* dst;
  int64_t ldb, K, Kpad, Jn, Npad;
  int64_t start;   // first block
};
struct PrepBatch {
  int n, type;
  PrepJob job[2];
};
constexpr int kPrepPairs = 4;   // pairs of a thread

__global__ void __launch_bounds__(256) tcg_prepare_kernel(const __grid_constant__ PrepBatch b) {
  const PrepJob& j = b.job[b.n > 1 && (int64_t)blockIdx.x >= b.job[1].start ? 1 : 0];
  const int64_t half = j.Kpad / 2, pairs = j.Npad * half;
  const int64_t e0 = ((int64_t)blockIdx.x - j.start) * (256 * kPrepPairs) + threadIdx.x;
#pragma unroll
  for (int u = 0; u < kPrepPairs; ++u) {
    const int64_t e = e0 + u * 256;
    if (e >= pairs) return;
    const int64_t row = e / half, k = 2 * (e - row * half);
    const bool a = row < j.Jn && k < j.K, c = row < j.Jn && k + 1 < j.K;
    const int64_t at = row * j.ldb + k;
    uint32_t* out = reinterpret_cast<uint32_t*>(j.dst) + e;
    if (b.type == 2) {
      const uint16_t* s = (const uint16_t*)j.src;
      *out = (a ? (uint32_t)s[at] : 0u) | ((c ? (uint32_t)s[at + 1] : 0u) << 16);
    } else {
      const float* s = (const float*)j.src;
      uint32_t w[3];
      cut3(a ? s[at] : 0.f, c ? s[at + 1] : 0.f, w);
#pragma unroll
      for (int q = 0; q < 3; ++q) out[q * pairs] = w[q];
    }
  }
}

// Sums the pieces of the row tiles that more than one CTA worked on.
__global__ void __launch_bounds__(256) tcg_pieces_kernel(const float* part, int64_t I, int nI,
                                                         int nkt, int G, int Npad, float* C) {
  const int it = blockIdx.x;
  const int64_t total = (int64_t)nI * nkt;
  auto owner = [&](int64_t u) { return (int)(((u + 1) * G - 1) / total); };
  const int c0 = owner((int64_t)it * nkt), c1 = owner((int64_t)(it + 1) * nkt - 1);
  if (c0 == c1) return;
  const int64_t rows = min((int64_t)kTileM, I - (int64_t)it * kTileM);
  const int n4 = (int)(rows * Npad / 4);
  const int64_t tile4 = (int64_t)kTileM * Npad / 4;
  // only the first CTA's range can begin in an earlier tile
  const float4* p4 = reinterpret_cast<const float4*>(part);
  const float4* f4 = p4 + (int64_t)(2 * c0 + ((int)(total * c0 / G / nkt) < it)) * tile4;
  float4* o4 = reinterpret_cast<float4*>(C) + (int64_t)it * tile4;
  for (int e = blockIdx.y * 256 + threadIdx.x; e < n4; e += gridDim.y * 256) {
    float4 a = f4[e];
#pragma unroll 4
    for (int c = c0 + 1; c <= c1; ++c) {
      const float4 v = p4[(int64_t)(2 * c) * tile4 + e];
      a.x += v.x;
      a.y += v.y;
      a.z += v.z;
      a.w += v.w;
    }
    o4[e] = a;
  }
}

struct TcgGeometry {
  int NS, KT, Npad, nI, nkt, stages, grid;
  int64_t Kpad, b_bytes, p_bytes;
  size_t smem;
};

static TcgGeometry tcg_geometry(const TcGemm& g, int sms) {
  TcgGeometry o;
  o.NS = g.type == 2 ? 1 : 3;
  o.KT = g.type == 2 ? 128 : 64;
  o.Npad = (int)round_up(g.Jn, 16);
  o.nI = (int)ceil_div(g.I, (int64_t)kTileM);
  o.nkt = (int)ceil_div(g.K, (int64_t)o.KT);
  o.Kpad = (int64_t)o.nkt * o.KT;
  const int64_t stage = (int64_t)o.NS * (128 * o.KT * 2 + (int64_t)o.Npad * o.KT * 2);
  o.stages = (int)std::min<int64_t>(kTcgMaxStages, (kSmemBudget - 1024) / stage);
  o.smem = (size_t)(1024 + o.stages * stage);
  // at least two tiles per CTA: a shorter range is mostly fill and drain
  o.grid = (int)std::max<int64_t>(1, std::min<int64_t>((int64_t)o.nI * o.nkt / 2, sms));
  o.b_bytes = round_up((int64_t)o.NS * o.Npad * o.Kpad * 2, 256);
  o.p_bytes = (int64_t)2 * sms * kTileM * o.Npad * 4;   // (as for a full grid: grows with the shape only)
  return o;
}

template <typename T, bool MN, bool VEC, int NW>
static ttnn_status tcg_launch(const TcgGeometry& o, const CUtensorMap& mB, const TcgParams& p,
                              cudaStream_t st) {
  constexpr int slot = 4 + (NW > 64 ? 8 : 0) + (sizeof(T) == 4 ? 4 : 0) + (MN ? 2 : 0) + (VEC ? 1 : 0);
  TTNN_TRY(smem_limit_once((const void*)tcg_kernel<T, MN, VEC, NW>, slot));
  tcg_kernel<T, MN, VEC, NW><<<o.grid, tcg_threads<NW>(), o.smem, st>>>(mB, p);
  return check_launch("tcg_kernel");
}

template <typename T, bool VEC, int NW>
static ttnn_status tcg_major(bool mn, const TcgGeometry& o, const CUtensorMap& mB,
                             const TcgParams& p, cudaStream_t st) {
  return mn ? tcg_launch<T, true, VEC, NW>(o, mB, p, st) : tcg_launch<T, false, VEC, NW>(o, mB, p, st);
}

}  // namespace tc

bool tcg_supported(const TcGemm& g) {
  if (g.type == 0) return zgemm_supported(g);
  const int64_t lim = int64_t(1) << 31;
  if ((g.type != 1 && g.type != 2) || g.I < 1 || g.Jn < 1 || g.K < 1) return false;
  if (g.Jn > tc::kTcgMaxN || g.ldc != round_up(g.Jn, 16)) return false;
  // 32-bit tile counts and TMA coordinates
  return g.I < lim - 256 && g.K < lim - 256;
}

int64_t tcg_prep_bytes(const TcGemm& g) {
  return g.type == 0 ? zgemm_prep_bytes(g) : tc::tcg_geometry(g, 1).b_bytes;
}

ttnn_status tcg_prepare(const TcGemm* g, int n, void* const* dst, cudaStream_t st) {
  using namespace tc;
  if (g[0].type == 0) return zgemm_prepare(g, n, dst, st);
  PrepBatch pb;
  pb.n = n;
  pb.type = g[0].type;
  int64_t blocks = 0;
  for (int k = 0; k < n; ++k) {
    const TcgGeometry o = tcg_geometry(g[k], 1);
    PrepJob& j = pb.job[k];
    j.src = g[k].B;
    j.dst = (uint16_t*)dst[k];
    j.ldb = g[k].ldb;
    j.K = g[k].K;
    j.Kpad = o.Kpad;
    j.Jn = g[k].Jn;
    j.Npad = o.Npad;
    j.start = blocks;
    blocks += ceil_div(j.Npad * j.Kpad / 2, (int64_t)256 * kPrepPairs);
  }
  if (blocks >= (int64_t(1) << 31)) {
    set_error("tensor-core GEMM: operand too large");
    return TTNN_EUNSUPPORTED;
  }
  tcg_prepare_kernel<<<(unsigned)blocks, 256, 0, st>>>(pb);
  return check_launch("tcg_prepare_kernel");
}

static ttnn_status launch_tcg_one(const TcGemm& g, const void* prep, void* pieces, int sms, int* err,
                                  uint64_t wait_ns, cudaStream_t st) {
  using namespace tc;
  const TcgGeometry o = tcg_geometry(g, sms);
  CUtensorMap mB;
  TTNN_TRY(encode_map(&mB, prep, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, o.Kpad, (int64_t)o.NS * o.Npad,
                      64u, (uint32_t)o.Npad, CU_TENSOR_MAP_SWIZZLE_128B));
  TcgParams p;
  p.A = g.A;
  p.lda = g.lda;
  p.I = g.I;
  p.K = g.K;
  p.nI = o.nI;
  p.nkt = o.nkt;
  p.Npad = o.Npad;
  p.stages = o.stages;
  // Chain of leading products per drain: 128 k (8 MMAs).  Long binary32
  // reductions take 256: their sums err less than the SIMT GEMM's by more
  // than the longer chain adds (64^4 x 8 slab: 4.2e-7 against 9.8e-7; short
  // ones would lose that margin), and the drains cost 10 % of the time.
  p.group = g.type == 2 ? 1 : g.K >= 2048 ? 4 : 2;
  p.C = (float*)g.C;
  p.part = (float*)pieces;
  p.err = err;
  p.wait_ns = wait_ns;
  const int64_t inner = g.mn ? g.I : g.K;
  const int pair = g.type == 2 ? 4 : 8;
  const bool vec = inner % 2 == 0 && g.lda % 2 == 0 && (uintptr_t)g.A % pair == 0;
  const bool mn = g.mn != 0, wide = o.Npad > 64;
  if (g.type == 2 && vec)
    TTNN_TRY(wide ? tcg_major<uint16_t, true, kTcgMaxN>(mn, o, mB, p, st)
                  : tcg_major<uint16_t, true, 64>(mn, o, mB, p, st));
  else if (g.type == 2)
    TTNN_TRY(wide ? tcg_major<uint16_t, false, kTcgMaxN>(mn, o, mB, p, st)
                  : tcg_major<uint16_t, false, 64>(mn, o, mB, p, st));
  else if (vec)
    TTNN_TRY(wide ? tcg_major<float, true, kTcgMaxN>(mn, o, mB, p, st)
                  : tcg_major<float, true, 64>(mn, o, mB, p, st));
  else
    TTNN_TRY(wide ? tcg_major<float, false, kTcgMaxN>(mn, o, mB, p, st)
                  : tcg_major<float, false, 64>(mn, o, mB, p, st));
  if (o.grid == 1) return TTNN_OK;
  const int per = (int)std::max<int64_t>(1, std::min<int64_t>(8, 608 / std::max(1, o.nI)));
  tcg_pieces_kernel<<<dim3((unsigned)o.nI, (unsigned)per), 256, 0, st>>>(
      (const float*)pieces, g.I, o.nI, o.nkt, o.grid, o.Npad, (float*)g.C);
  return check_launch("tcg_pieces_kernel");
}

ttnn_status launch_tcg(const TcGemm* g, int n, int sms, int* err, uint64_t wait_ns, void* ws,
                       int64_t ws_bytes, cudaStream_t st, bool dry, int64_t* need) {
  int64_t b_bytes = 0, p_bytes = 0;
  void* dst[2] = {nullptr, nullptr};
  TcGemm todo[2];
  int nt = 0;
  char* w = (char*)ws + (256 - ((uintptr_t)ws & 255)) % 256;
  for (int k = 0; k < n; ++k) {
    // the products run in order and share the room of their pieces
    p_bytes = std::max(p_bytes, g[k].type == 0 ? zgemm_piece_bytes(g[k], sms)
                                               : tc::tcg_geometry(g[k], sms).p_bytes);
    if (g[k].prep) continue;
    todo[nt] = g[k];
    dst[nt++] = w + b_bytes;
    b_bytes += tcg_prep_bytes(g[k]);
  }
  if (dry) {
    *need = b_bytes + p_bytes + 256;
    return TTNN_OK;
  }
  if (w + b_bytes + p_bytes > (char*)ws + ws_bytes) {
    set_error("tensor-core GEMM: workspace too small");
    return TTNN_ENOMEM;
  }
  if (nt > 0) TTNN_TRY(tcg_prepare(todo, nt, dst, st));
  nt = 0;
  for (int k = 0; k < n; ++k) {
    const void* prep = g[k].prep ? g[k].prep : dst[nt++];
    TTNN_TRY(g[k].type == 0 ? launch_zgemm(g[k], prep, w + b_bytes, sms, err, wait_ns, st)
                            : launch_tcg_one(g[k], prep, w + b_bytes, sms, err, wait_ns, st));
  }
  return TTNN_OK;
}

}  // namespace ttnn
