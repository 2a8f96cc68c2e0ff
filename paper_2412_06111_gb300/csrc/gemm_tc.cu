// GEMM on the tcgen05 tensor cores with the large operand loaded by converter
// warps instead of TMA, for first-level products of tensors whose rows TMA
// cannot address (a stride that is not a multiple of 16 bytes) and of
// binary32 boxes.  The SIMT GEMM these took before ran at 12.5 TFLOP/s of the
// 80 the FMA pipes have; here the tensor is read at HBM speed and the
// products run on the tensor cores.
//
// Precision.  bfloat16 operands are multiplied as they are.  A binary32
// operand is cut into three bfloat16 pieces, the second and third scaled by 2^6
// and 2^12, which give every entry from 2^-122 in magnitude on exactly (below, a
// multiple of 2^-145 next to it; cut3).  The six products down to 2^-16 of the
// leading one are formed, the other three (2^-24 and below, of either sign) are
// left out.  The tensor core truncates when it adds to
// its binary32 accumulator, so chains are short: the leading products of 32 to
// 256 k go into one accumulator, those of each lower order into another, and the
// epilogue warps add them to registers with rounding to nearest.  The pieces
// of B sit below one another in shared memory, so piece i of A meets all the
// pieces of B it is multiplied with in one MMA of up to three times the
// columns: the MMAs are bound by reading their operands from shared memory
// (about 100 cycles for 128 x 64 x 16), and A is read three times per k step
// instead of six.
//
// Warp roles: warp 0 copies B tiles by TMA, warp 1 owns TMEM and issues the
// MMAs, the next 8 drain accumulators (TMEM lane quarter = warp % 4), the
// last 16 load, convert and store A tiles (128-byte swizzle).  Every wait is
// bounded; on expiry the kernel sets an error bit, drains its own copies and
// MMAs, frees TMEM and returns.
#include <cuda_bf16.h>

#include <algorithm>
#include <cfloat>
#include <type_traits>

#include "gemm_tc.cuh"
#include "tc_ptx.cuh"

namespace ttnn {
namespace tc {

constexpr int kTcgMaxN = 80;      // columns of a product
constexpr int kTcgConv = 16;      // converter warps (8 left the latency of the loads bare: twice the time)
// Epilogue warps: two per lane quarter, a half of the columns each (one per
// quarter holds twice the sums and spills: 64^5 bfloat16 514 against 509 us, a
// rank-200 TTN update 659 against 650, an 8 x 64^4 binary32 slab 365 against 367).
constexpr int kTcgEpi = 8;
constexpr int kTcgThreads = 32 * (2 + kTcgEpi + kTcgConv);
constexpr int kTcgMaxStages = 6;

struct TcgProb {
  CUtensorMap mapB;
  const void* A;
  int64_t lda, I, K;
  float* C;
  int64_t ldc, unit0;    // first (row tile, k tile) of the product in the launch
  int nkt, tile0;        // k tiles, first row tile in the launch
  int chain;             // MMAs (of 16 k) per drain of the accumulators: 2 (not bfloat16), 8 or 16
  int trans;
};
struct TcgParams {
  int n, tiles;          // products, row tiles of all of them
  int Npad, stages;
  int64_t units;         // (row tile, k tile) pairs of all of them
  float* part;           // pieces [2 grid][128][Npad]
  int* err;
  uint64_t wait_ns;
  TcgProb prob[kTcgBatch];
};
static_assert(sizeof(TcgParams) <= 4096, "a launch's products travel in the kernel parameters");

// x 2^e for |e| < 252 (one rounding more where the result is subnormal).
__device__ __forceinline__ float scale2(float x, int e) {
  return x * __int_as_float((127 + e / 2) << 23) * __int_as_float((127 + e - e / 2) << 23);
}

// The product of row tile `it` of the launch.
__device__ __forceinline__ int tcg_prob(const TcgParams& p, int it) {
  int q = 0;
  while (q + 1 < p.n && it >= p.prob[q + 1].tile0) ++q;
  return q;
}
// The row tile that holds unit u.
__device__ __forceinline__ int tcg_tile(const TcgParams& p, int64_t u) {
  int q = 0;
  while (q + 1 < p.n && u >= p.prob[q + 1].unit0) ++q;
  return p.prob[q].tile0 + (int)((u - p.prob[q].unit0) / p.prob[q].nkt);
}
// The first unit of row tile `it` (of product q).
__device__ __forceinline__ int64_t tcg_unit(const TcgParams& p, int q, int it) {
  return p.prob[q].unit0 + (int64_t)(it - p.prob[q].tile0) * p.prob[q].nkt;
}

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
template <>
struct Form<double> {   // rounded to binary32 on the way
  static constexpr int NS = 3, KT = 64, NACC = 3, NG = 1;
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

template <bool VEC>
struct Pair<double, VEC> {
  double x, y;
  __device__ void load(const double* p, bool a, bool b) {
    if (VEC) {
      const double2 v = a ? __ldg(reinterpret_cast<const double2*>(p)) : make_double2(0., 0.);
      x = v.x;
      y = v.y;
    } else {
      x = a ? __ldg(p) : 0.;
      y = b ? __ldg(p + 1) : 0.;
    }
  }
};

// The three pieces of two binary32 values, packed (x in the low half).  The
// first is cut toward zero, so that no finite value overflows; the second is
// rounded, which leaves the third either sign: the piece products left out
// then average to nothing (a 200-rank tree's Psi erred by 6.2e-7 with both cut
// toward zero, 4.8e-7 so).  The first piece of an infinity or NaN is it, its
// other pieces are NaN: the sums of lower order are NaN then, and the epilogue
// leaves what the leading products give, as binary32 multiply-adds would.
//
// bfloat16 ends at 2^-133: unscaled, the pieces of a binary32 entry below 2^-110
// lose its low bits (entries of 1e-35: 4.4e-6 off).  With piece i times 2^(6 i) the
// products of order o = i + j are 2^(6 o) too large, which the epilogue takes
// back; 2^6 is the most for which the sums of order 1 (two products below 2^-7
// of the leading one each) cannot overflow before those of order 0.  (The
// multiplications cost a binary32 box of 8 x 64^4 20 of 371 us; packed in pairs
// they cost 36, in spills.)
constexpr float kPieceScale = 64.f;
__device__ __forceinline__ void cut3(float x, float y, uint32_t* w) {
  // (not a cut of the bits: a NaN may have all of its in the lower half)
  asm("cvt.rz.bf16x2.f32 %0, %1, %2;" : "=r"(w[0]) : "f"(y), "f"(x));
  x = (x - __uint_as_float(w[0] << 16)) * kPieceScale;
  y = (y - __uint_as_float(w[0] & 0xFFFF0000u)) * kPieceScale;
  const __nv_bfloat162 v = __floats2bfloat162_rn(x, y);
  w[1] = *reinterpret_cast<const uint32_t*>(&v);
  x = (x - __uint_as_float(w[1] << 16)) * kPieceScale;
  y = (y - __uint_as_float(w[1] & 0xFFFF0000u)) * kPieceScale;
  w[2] = __byte_perm(__float_as_uint(x), __float_as_uint(y), 0x7632);
}

// a s + b and a + b of two columns in one instruction each.
__device__ __forceinline__ float2 fma2(float2 a, float s, float2 b) {
  float2 r;
  asm("{\n\t.reg .b64 a, b, s;\n\tmov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %5};\n\tmov.b64 s, {%6, %6};\n\t"
      "fma.rn.f32x2 a, a, s, b;\n\tmov.b64 {%0, %1}, a;\n\t}\n"
      : "=f"(r.x), "=f"(r.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(s));
  return r;
}
__device__ __forceinline__ float2 add2(float2 a, float2 b) {
  float2 r;
  asm("{\n\t.reg .b64 a, b;\n\tmov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %5};\n\t"
      "add.rn.f32x2 a, a, b;\n\tmov.b64 {%0, %1}, a;\n\t}\n"
      : "=f"(r.x), "=f"(r.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return r;
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

template <typename T, bool MN, bool VEC>
__global__ void __launch_bounds__(kTcgThreads, 1)
    tcg_kernel(const __grid_constant__ TcgParams p) {
  using F = Form<T>;
  constexpr int NW = kTcgMaxN / 2;               // columns an epilogue thread holds sums of
  constexpr int NS = F::NS, KT = F::KT, NACC = F::NACC;
  constexpr int R = MN ? KT : kTileM;            // tile rows in memory order
  constexpr int CB = MN ? 2 : KT / 64;           // 64-column boxes of a row
  constexpr int NG = F::NG;                      // converter groups, a tile each in turn
  constexpr int NCW = kTcgConv / NG;             // warps of a group
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
  // The (row tile, k tile) units of all products, in order, are cut into
  // gridDim.x even ranges, one per CTA.  Row tiles within one range go to C;
  // only the first and the last of a range can be pieces of a tile (slots 2 c
  // and 2 c + 1 of CTA c), which are summed afterwards in CTA order.
  const int64_t u0 = p.units * blockIdx.x / gridDim.x, u1 = p.units * (blockIdx.x + 1) / gridDim.x;
  const int i0 = tcg_tile(p, u0), i1 = u1 > u0 ? tcg_tile(p, u1 - 1) + 1 : i0;

  if (threadIdx.x == 0) {
    abort_flag = 0;
    for (int s = 0; s < S; ++s) {
      mbar_init(smem_u32(&bar_a[s]), NCW);
      mbar_init(smem_u32(&bar_b[s]), 1);
      mbar_init(smem_u32(&bar_empty[s]), 1);
    }
    for (int k = 0; k < 2; ++k) {
      mbar_init(smem_u32(&bar_full[k]), 1);
      mbar_init(smem_u32(&bar_free[k]), kTcgEpi);
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

  // this CTA's k tiles of row tile `it`, and its product
  auto range = [&](int it, int* kt0, int* kt1) {
    const int q = tcg_prob(p, it);
    const int64_t r = tcg_unit(p, q, it);
    *kt0 = (int)(max(u0, r) - r);
    *kt1 = (int)(min(u1, r + p.prob[q].nkt) - r);
    return q;
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
        const CUtensorMap* mapB = &p.prob[range(it, &kt0, &kt1)].mapB;
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
              tma_2d(sb + s * b_piece + h * (b_piece / (KT / 64)), mapB, kt * KT + h * 64,
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
        const int chain = p.prob[range(it, &kt0, &kt1)].chain;
        int steps = 0;      // MMAs deep the accumulators at hand are
        for (int kt = kt0; kt < kt1; ++kt) {
          ok = mbar_wait(smem_u32(&bar_a[stage]), ph, &abort_flag, p.wait_ns) &&
               mbar_wait(smem_u32(&bar_b[stage]), ph, &abort_flag, p.wait_ns);
          if (!ok) break;
          const uint32_t sa = base + stage * stage_bytes;
          const uint32_t sb = sa + NS * kPiece;
          // the MMAs of `n` k steps from k0 on (unrolled: this thread's issue
          // rate bounds the kernel when each drain is short)
          auto issue = [&](auto first, auto count) {
            constexpr int k0 = decltype(first)::value, n = decltype(count)::value;
            if (steps == 0) {
              ok = mbar_wait(smem_u32(&bar_free[buf]), fph, &abort_flag, p.wait_ns);
              if (!ok) return;
            }
            fence_after();
            const uint32_t d = tmem + buf * NACC * p.Npad;
            const uint64_t a = sdesc(sa, MN ? kBox : 16, 1024), b = sdesc(sb, 16, 1024);
#pragma unroll
            for (int ia = 0; ia < NS; ++ia) {
              // piece ia of A against pieces 0 .. NS - 1 - ia of B: orders ia .. NS - 1
              const uint32_t id = idesc_bf16(kTileM, (NS - ia) * p.Npad, MN);
#pragma unroll
              for (int kk = k0; kk < k0 + n; ++kk) {
                mma_bf16(d + ia * p.Npad,
                         sdesc_at(a, ia * kPiece + (MN ? kk * 2048 : (kk >> 2) * kBox + (kk & 3) * 32)),
                         sdesc_at(b, (kk >> 2) * (p.Npad * 128) + (kk & 3) * 32), id,
                         kk > k0 || ia > 0 || steps > 0);
              }
            }
            steps += n;
            if (steps >= chain || (kt + 1 == kt1 && k0 + n == KT / 16)) {
              mma_commit(smem_u32(&bar_full[buf]));
              buf ^= 1;
              if (buf == 0) fph ^= 1;
              steps = 0;
            }
          };
          if (chain >= KT / 16) {
            issue(std::integral_constant<int, 0>(), std::integral_constant<int, KT / 16>());
          } else if constexpr (NS > 1) {   // chains of two
            issue(std::integral_constant<int, 0>(), std::integral_constant<int, 2>());
            if (ok) issue(std::integral_constant<int, 2>(), std::integral_constant<int, 2>());
          }
          if (!ok) break;
          mma_commit(smem_u32(&bar_empty[stage]));
          if (++stage == S) {
            stage = 0;
            ph ^= 1;
          }
        }
      }
      if (!ok) {
        abort_flag = 1;
        atomicOr(p.err, 4);
      }
      mma_commit(smem_u32(&bar_done));
    }
  } else if (warp >= 2 + kTcgEpi) {
    // ---------------- converters ----------------
    const int cw = (warp - 2 - kTcgEpi) % NCW, grp = (warp - 2 - kTcgEpi) / NCW;
    int stage = 0;
    uint32_t ph = 0;
    bool ok = true;
    // v holds a tile's pairs; each is reloaded for the next tile as soon as
    // it is stored, so a whole tile of loads is in flight per warp
    Pair<T, VEC> v[NP];
    int it = i0, kt = 0, kt1 = 0;
    const T* A = nullptr;       // of the product at hand
    int64_t lda = 0, rows = 0, cols = 0;
    int tile0 = 0;
    const T* src = nullptr;
    int nrow = 0, ncol = 0;     // valid rows of the warp, valid columns from the lane's on
    auto aim = [&]() {
      const int64_t k0 = kt * (int64_t)KT, j0 = (it - tile0) * (int64_t)kTileM;
      const int64_t r0 = (MN ? k0 : j0) + cw * RW, c0 = (MN ? j0 : k0) + 2 * lane;
      src = A + r0 * lda + c0;
      nrow = (int)max((int64_t)0, min((int64_t)RW, rows - r0));
      ncol = (int)max((int64_t)0, min((int64_t)256, cols - c0));
    };
    // every pair of the warp inside the operand: no bounds on the loads
    auto interior = [&]() {
      return __all_sync(0xffffffffu, nrow == RW && ncol > (CB - 1) * 64 + 1);
    };
    auto load = [&](int q, bool all) {
      const int rr = q / CB, c = (q % CB) * 64;
      v[q].load(src + (int64_t)rr * lda + c, all || (rr < nrow && c < ncol),
                all || (rr < nrow && c + 1 < ncol));
    };
    auto enter = [&]() {
      const TcgProb& b = p.prob[range(it, &kt, &kt1)];
      A = (const T*)b.A;
      lda = b.lda;
      rows = MN ? b.K : b.I;
      cols = MN ? b.I : b.K;
      tile0 = b.tile0;
    };
    // on by n tiles of this CTA's range
    auto advance = [&](int n) {
      kt += n;
      while (it < i1 && kt >= kt1) {
        n = kt - kt1;
        if (++it < i1) {
          enter();
          kt += n;
        }
      }
    };
    if (it < i1) {
      enter();
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
          cut3((float)v[q].x, (float)v[q].y, w);
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
    // ---------------- epilogue ----------------
    const int q = warp & 3;
    const int cn = p.Npad / 2, cb = (warp - 2) / 4 * cn;   // this warp's columns (a multiple of 8)
    const uint32_t lane_off = (uint32_t)(32 * q) << 16;
    int buf = 0;
    uint32_t fph = 0;
    bool ok = true;
    for (int it = i0; it < i1 && ok; ++it) {
      int kt0, kt1;
      const TcgProb& b = p.prob[range(it, &kt0, &kt1)];
      float acc[NW];
#pragma unroll
      for (int c = 0; c < NW; ++c) acc[c] = 0.f;
      const int drains = ((kt1 - kt0) * (KT / 16) + b.chain - 1) / b.chain;
      for (int g = 0; g < drains; ++g) {
        ok = mbar_wait(smem_u32(&bar_full[buf]), fph, &abort_flag, p.wait_ns);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        fence_after();
        const uint32_t d = tmem + lane_off + buf * NACC * p.Npad + cb;
#pragma unroll
        for (int cg = 0; cg < NW; cg += 8) {
          if (cg >= cn) continue;
          uint32_t x[NACC][8];
#pragma unroll
          for (int o = 0; o < NACC; ++o) tmem_ld8(d + o * p.Npad + cg, x[o]);
          tmem_wait_ld();
#pragma unroll
          for (int c = 0; c < 8; c += 2) {
            float2 v = make_float2(__uint_as_float(x[NACC - 1][c]), __uint_as_float(x[NACC - 1][c + 1]));
#pragma unroll
            for (int o = NACC - 2; o >= 0; --o) {
              // sums without the leading products are NaN wherever those are
              // not finite: a finite value in their place leaves the result
              if (o == 0) v = make_float2(fmaxf(v.x, -FLT_MAX), fmaxf(v.y, -FLT_MAX));
              v = fma2(v, 1.f / kPieceScale, make_float2(__uint_as_float(x[o][c]), __uint_as_float(x[o][c + 1])));
            }
            const float2 a = add2(make_float2(acc[cg + c], acc[cg + c + 1]), v);
            acc[cg + c] = a.x;
            acc[cg + c + 1] = a.y;
          }
        }
        fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&bar_free[buf]));
        buf ^= 1;
        if (buf == 0) fph ^= 1;
      }
      if (!ok) break;
      const bool whole = kt0 == 0 && kt1 == b.nkt;
      const int64_t row = (int64_t)(it - b.tile0) * kTileM + 32 * q + lane;
      if (row < b.I && whole && b.trans) {
        float* out = b.C + cb * b.ldc + row;
#pragma unroll
        for (int c = 0; c < NW; ++c)
          if (c < cn) out[(int64_t)c * b.ldc] = acc[c];
      } else if (row < b.I) {
        float* dst = whole ? b.C + row * b.ldc
                           : p.part + ((int64_t)(2 * blockIdx.x + (it > i0)) * kTileM + 32 * q + lane) * p.Npad;
        float4* out = reinterpret_cast<float4*>(dst + cb);
#pragma unroll
        for (int c = 0; c < NW / 4; ++c)
          if (4 * c < cn) out[c] = make_float4(acc[4 * c], acc[4 * c + 1], acc[4 * c + 2], acc[4 * c + 3]);
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
  TcCols c[2];
  uint16_t* dst;
  int32_t* shift;
  int64_t K, Kpad;
  int nb, Npad, bf16, start;   // start: first block
};
struct PrepBatch {
  int n;
  PrepJob job[kTcgBatch];
};
constexpr int kPrepRows = 8;   // rows of a thread

// The powers of two that column j of a Khatri-Rao operand loses.  Its factors
// are sketches and environments of a network, of any size: their product may
// leave binary32 although its sum against the core is representable.  The
// largest magnitudes of the factors, 2^e0 and 2^e1 (not above e0 + 1, e1 + 1),
// are brought to 2^32 (2^-32) each if e0 + e1 > 64 (< -64), else left alone:
// what then over- or underflows in the sum against binary32 entries does so in
// the result.  Blocks: a column (x) of a job (y).
__global__ void __launch_bounds__(256) tcg_range_kernel(const __grid_constant__ PrepBatch b) {
  pdl_begin();
  const PrepJob& j = b.job[blockIdx.y];
  const TcCols& c = j.c[0];
  const int col = blockIdx.x, warp = threadIdx.x >> 5;
  if (!j.shift || col >= j.Npad) return;
  __shared__ uint32_t big[2][8];
#pragma unroll
  for (int f = 0; f < 2; ++f) {
    uint32_t m = 0u;
    if (col < c.n)
      for (int64_t i = threadIdx.x; i < c.krn[f]; i += 256)
        m = max(m, __float_as_uint(c.kr[f][i * c.ki[f] + col * c.kj[f]]) & 0x7FFFFFFFu);
    m = __reduce_max_sync(0xffffffffu, m);
    if ((threadIdx.x & 31) == 0) big[f][warp] = m;
  }
  __syncthreads();
  if (threadIdx.x != 0) return;
  int e[2];
  for (int f = 0; f < 2; ++f) {
    uint32_t m = 0u;
    for (int w = 0; w < 8; ++w) m = max(m, big[f][w]);
    // (subnormal: not above 2^(e + 1); 0: any; not finite: 128)
    e[f] = m < 0x00800000u ? m ? -118 - __clz(m) : 0 : (int)(m >> 23) - 127;
  }
  const int to = e[0] + e[1] > 64 ? 32 : -32;
  const bool off = e[0] + e[1] > 64 || e[0] + e[1] < -64;
  j.shift[2 * col] = off ? e[0] - to : 0;
  j.shift[2 * col + 1] = off ? e[1] - to : 0;
}

__device__ __forceinline__ float prep_value(const TcCols& c, const int32_t* shift, int64_t j, int64_t k) {
  if (c.nkr == 0) return ((const float*)c.p)[j * c.sj + k * c.sk];
  if (shift && (shift[2 * j] | shift[2 * j + 1])) {
    const uint32_t d0 = (uint32_t)k / (uint32_t)c.krn[1], d1 = (uint32_t)k - d0 * (uint32_t)c.krn[1];
    return scale2(c.kr[0][(int64_t)d0 * c.ki[0] + j * c.kj[0]], -shift[2 * j]) *
           scale2(c.kr[1][(int64_t)d1 * c.ki[1] + j * c.kj[1]], -shift[2 * j + 1]);
  }
  float v = 1.f;
  uint32_t rem = (uint32_t)k;
#pragma unroll
  for (int f = 3; f >= 0; --f) {
    if (f >= c.nkr) continue;
    const uint32_t q = rem / (uint32_t)c.krn[f];
    v *= c.kr[f][(int64_t)(rem - q * (uint32_t)c.krn[f]) * c.ki[f] + j * c.kj[f]];
    rem = q;
  }
  return v;
}

// Blocks of a job: 256 pairs of k by kPrepRows rows.
__global__ void __launch_bounds__(256) tcg_prepare_kernel(const __grid_constant__ PrepBatch b) {
  int at = 0;
  while (at + 1 < b.n && (int)blockIdx.x >= b.job[at + 1].start) ++at;
  const PrepJob& j = b.job[at];
  const int half = (int)(j.Kpad / 2), kblocks = (half + 255) / 256;
  const int blk = (int)blockIdx.x - j.start;
  const int kp = blk % kblocks * 256 + (int)threadIdx.x, row0 = blk / kblocks * kPrepRows;
  if (kp >= half) return;
  const int64_t k = 2 * (int64_t)kp, pairs = (int64_t)j.Npad * half;
#pragma unroll
  for (int u = 0; u < kPrepRows; ++u) {
    int row = row0 + u;
    uint32_t* out = reinterpret_cast<uint32_t*>(j.dst) + (int64_t)row * half + kp;
    const bool second = row >= j.c[0].n && j.nb > 1;
    const TcCols& c = j.c[second ? 1 : 0];
    if (second) row -= j.c[0].n;
    const bool in = row < c.n && k < j.K, in1 = in && k + 1 < j.K;
    if (j.bf16) {
      const uint16_t* s = (const uint16_t*)c.p + row * c.sj + k * c.sk;
      *out = (in ? (uint32_t)s[0] : 0u) | ((in1 ? (uint32_t)s[c.sk] : 0u) << 16);
    } else {
      uint32_t w[3];
      cut3(in ? prep_value(c, j.shift, row, k) : 0.f, in1 ? prep_value(c, j.shift, row, k + 1) : 0.f, w);
#pragma unroll
      for (int q = 0; q < 3; ++q) out[q * pairs] = w[q];
    }
  }
}

// Sums the pieces of the row tiles that more than one CTA worked on: block c
// takes the tile in which CTA c's range begins, if it is the first to begin
// inside it.
__global__ void __launch_bounds__(256) tcg_pieces_kernel(const __grid_constant__ TcgParams p, int G) {
  const int c = blockIdx.x + 1;
  const int64_t u = p.units * c / G, before = p.units * (c - 1) / G;
  const int it = tcg_tile(p, u), q = tcg_prob(p, it);
  const TcgProb& b = p.prob[q];
  const int64_t first = tcg_unit(p, q, it);
  if (u == first || before > first) return;
  const int c0 = c - 1, c1 = (int)(((first + b.nkt) * G - 1) / p.units);
  const int64_t r0 = (int64_t)(it - b.tile0) * kTileM;
  const int rows = (int)min((int64_t)kTileM, b.I - r0);
  const int64_t tile = (int64_t)kTileM * p.Npad;
  // only the first CTA's range can begin in an earlier tile
  const float* p0 = p.part + (2 * c0 + (before < first)) * tile;
  const int per = p.Npad / 4;
  for (int e = blockIdx.y * 256 + threadIdx.x; e < rows * per; e += gridDim.y * 256) {
    // transposed results: consecutive threads take consecutive rows
    const int r = b.trans ? e % rows : e / per, c4 = b.trans ? e / rows : e % per;
    const int64_t at = (int64_t)r * p.Npad + 4 * c4;
    float4 a = *reinterpret_cast<const float4*>(p0 + at);
#pragma unroll 4
    for (int d = c; d <= c1; ++d) {
      const float4 v = *reinterpret_cast<const float4*>(p.part + (int64_t)(2 * d) * tile + at);
      a.x += v.x;
      a.y += v.y;
      a.z += v.z;
      a.w += v.w;
    }
    if (b.trans) {
      float* o = b.C + (int64_t)4 * c4 * b.ldc + r0 + r;
      o[0] = a.x;
      o[b.ldc] = a.y;
      o[2 * b.ldc] = a.z;
      o[3 * b.ldc] = a.w;
    } else {
      *reinterpret_cast<float4*>(b.C + (r0 + r) * b.ldc + 4 * c4) = a;
    }
  }
}

// Gives the powers of two of tcg_range_kernel back to the columns of C (column:
// x; rows: y; product: z).  A kernel of its own: in the epilogue it cost every
// product more than this launch (a rank-200 update 675 us against 656, 64^5 521
// against 516).
struct UnshiftBatch {
  struct {
    float* C;
    const int32_t* shift;
    int64_t I, si, sj;
    int Jn;
  } job[kTcgBatch];
};
__global__ void __launch_bounds__(256) tcg_unshift_kernel(const __grid_constant__ UnshiftBatch b) {
  pdl_begin();
  const auto& j = b.job[blockIdx.z];
  const int col = blockIdx.x;
  if (col >= j.Jn) return;
  const int e = j.shift[2 * col] + j.shift[2 * col + 1];
  if (e == 0) return;
  for (int64_t i = blockIdx.y * 256 + threadIdx.x; i < j.I; i += gridDim.y * 256) {
    float* c = j.C + i * j.si + col * j.sj;
    *c = scale2(*c, e);
  }
}

static int tcg_pieces_of(const TcGemm& g) { return g.type == 2 ? 1 : 3; }
static int tcg_kt(const TcGemm& g) { return g.type == 2 ? 128 : 64; }
static int tcg_npad(const TcGemm& g) { return (int)round_up(g.Jn, 16); }

template <typename T, bool MN, bool VEC>
static ttnn_status tcg_launch(const TcgParams& p, int grid, size_t smem, cudaStream_t st) {
  constexpr int kind = sizeof(T) == 2 ? 0 : sizeof(T) == 4 ? 1 : 2;
  constexpr int slot = 8 + kind * 4 + (MN ? 2 : 0) + (VEC ? 1 : 0);
  TTNN_TRY(smem_limit_once((const void*)tcg_kernel<T, MN, VEC>, slot));
  tcg_kernel<T, MN, VEC><<<grid, kTcgThreads, smem, st>>>(p);
  return check_launch("tcg_kernel");
}

template <typename T>
static ttnn_status tcg_form(bool vec, bool mn, const TcgParams& p, int grid, size_t smem,
                            cudaStream_t st) {
  if (mn) return vec ? tcg_launch<T, true, true>(p, grid, smem, st) : tcg_launch<T, true, false>(p, grid, smem, st);
  return vec ? tcg_launch<T, false, true>(p, grid, smem, st) : tcg_launch<T, false, false>(p, grid, smem, st);
}

// Pairs in one load need even extents and strides and an aligned base.
static bool tcg_vec(const TcGemm& g) {
  const int pair = g.type == 2 ? 4 : g.type == 1 ? 8 : 16;
  return (g.mn ? g.I : g.K) % 2 == 0 && g.lda % 2 == 0 && (uintptr_t)g.A % pair == 0;
}

// One launch: up to kTcgBatch products of one type, majorness, width and vec.
static ttnn_status tcg_batch(const TcGemm* const* g, int n, void* pieces, int sms, int* err,
                             uint64_t wait_ns, cudaStream_t st) {
  TcgParams p;
  const TcGemm& f = *g[0];
  const int NS = tcg_pieces_of(f), KT = tcg_kt(f);
  p.n = n;
  p.Npad = tcg_npad(f);
  p.tiles = 0;
  p.units = 0;
  for (int k = 0; k < n; ++k) {
    TcgProb& q = p.prob[k];
    const int64_t nI = ceil_div(g[k]->I, (int64_t)kTileM);
    q.nkt = (int)ceil_div(g[k]->K, (int64_t)KT);
    TTNN_TRY(encode_map(&q.mapB, g[k]->prep, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, (int64_t)q.nkt * KT,
                        (int64_t)NS * p.Npad, 64u, (uint32_t)p.Npad, CU_TENSOR_MAP_SWIZZLE_128B));
    q.A = g[k]->A;
    q.lda = g[k]->lda;
    q.I = g[k]->I;
    q.K = g[k]->K;
    q.C = (float*)g[k]->C;
    q.ldc = g[k]->ldc;
    q.trans = g[k]->trans;
    q.unit0 = p.units;
    q.tile0 = p.tiles;
    // Chain of leading products per drain: 8 MMAs (128 k).  Long binary32
    // reductions take 16: their sums err less than the SIMT GEMM's by more
    // than the longer chain adds (64^4 x 8 slab: 2.0e-7 against 6.5e-7; short
    // ones would lose that margin), and the drains cost 10 % of the time.
    q.chain = g[k]->chain ? g[k]->chain : f.type != 2 && g[k]->K >= 2048 ? 16 : 8;
    p.tiles += (int)nI;
    p.units += nI * q.nkt;
  }
  const int64_t stage = (int64_t)NS * (128 * KT * 2 + (int64_t)p.Npad * KT * 2);
  p.stages = (int)std::min<int64_t>(kTcgMaxStages, (kSmemBudget - 1024) / stage);
  p.part = (float*)pieces;
  p.err = err;
  p.wait_ns = wait_ns;
  const size_t smem = (size_t)(1024 + p.stages * stage);
  // at least two units per CTA: a shorter range is mostly fill and drain
  const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(p.units / 2, sms));
  const bool vec = tcg_vec(f), mn = f.mn != 0;
  if (f.type == 2) TTNN_TRY(tcg_form<uint16_t>(vec, mn, p, grid, smem, st));
  else if (f.type == 1) TTNN_TRY(tcg_form<float>(vec, mn, p, grid, smem, st));
  else TTNN_TRY(tcg_form<double>(vec, mn, p, grid, smem, st));
  if (grid > 1) {
    tcg_pieces_kernel<<<dim3((unsigned)(grid - 1), 4), 256, 0, st>>>(p, grid);
    TTNN_TRY(check_launch("tcg_pieces_kernel"));
  }
  UnshiftBatch u;
  int shifted = 0, most = 0;
  int64_t rows = 0;
  for (int k = 0; k < n; ++k) {
    const TcGemm& m = *g[k];
    if (!m.shift) continue;
    auto& j = u.job[shifted++];
    j.C = (float*)m.C;
    j.shift = m.shift;
    j.I = m.I;
    j.si = m.trans ? 1 : m.ldc;
    j.sj = m.trans ? m.ldc : 1;
    j.Jn = m.Jn;
    most = std::max(most, m.Jn);
    rows = std::max(rows, m.I);
  }
  if (shifted) {
    const unsigned by = (unsigned)std::min<int64_t>(ceil_div(rows, (int64_t)1024), 64);
    launch_pdl(tcg_unshift_kernel, dim3((unsigned)most, by, (unsigned)shifted), 256, 0, st, u);
    TTNN_TRY(check_launch("tcg_unshift_kernel"));
  }
  return TTNN_OK;
}

}  // namespace tc


bool tcg_supported(const TcGemm& g) {
  if (g.type == 0) return zgemm_supported(g);
  const int64_t lim = int64_t(1) << 31;
  if (g.type < 1 || g.type > 3 || g.I < 1 || g.Jn < 1 || g.K < 1) return false;
  if (g.Jn > tc::kTcgMaxN) return false;
  // a whole number of drains per tile or of tiles per drain (the issuer's two forms)
  if (g.chain != 0 && g.chain != 8 && g.chain != 16 && (g.chain != 2 || g.type == 2)) return false;
  if (g.shift && (g.nb != 1 || g.b[0].nkr != 2)) return false;
  // float4 rows of C
  if (!g.trans && (g.ldc < round_up(g.Jn, 16) || g.ldc % 4)) return false;
  // 32-bit tile counts (of kTcgBatch products) and TMA coordinates
  return g.I < lim - 256 && g.K < lim - 256;
}

int64_t tcg_prep_bytes(const TcGemm& g) {
  if (g.type == 0) return zgemm_prep_bytes(g);
  return round_up((int64_t)tc::tcg_pieces_of(g) * tc::tcg_npad(g) * round_up(g.K, (int64_t)tc::tcg_kt(g)) * 2, 256);
}

int64_t tcg_piece_bytes(const TcGemm& g, int sms) {
  return g.type == 0 ? zgemm_piece_bytes(g, sms) : (int64_t)2 * sms * tc::kTileM * tc::tcg_npad(g) * 4;
}

ttnn_status tcg_prepare(const TcGemm* g, int n, void* const* dst, cudaStream_t st) {
  using namespace tc;
  if (g[0].type == 0) return zgemm_prepare(g, n, dst, st);
  for (int k0 = 0; k0 < n; k0 += kTcgBatch) {
    PrepBatch pb;
    pb.n = std::min(n - k0, kTcgBatch);
    int64_t blocks = 0;
    int ranged = 0;   // columns of the widest operand that tcg_range_kernel looks over
    for (int k = 0; k < pb.n; ++k) {
      const TcGemm& m = g[k0 + k];
      PrepJob& j = pb.job[k];
      j.c[0] = m.b[0];
      j.c[1] = m.b[1];
      j.nb = m.nb;
      j.dst = (uint16_t*)dst[k0 + k];
      j.K = m.K;
      j.Kpad = round_up(m.K, (int64_t)tcg_kt(m));
      j.Npad = tcg_npad(m);
      j.bf16 = m.type == 2;
      j.shift = m.shift;
      if (m.shift) ranged = std::max(ranged, j.Npad);
      j.start = (int)blocks;
      blocks += ceil_div(j.Kpad / 2, (int64_t)256) * (j.Npad / kPrepRows);
      if (blocks >= (int64_t(1) << 31)) {
        set_error("tensor-core GEMM: operand too large");
        return TTNN_EUNSUPPORTED;
      }
    }
    if (ranged) {
      launch_pdl(tcg_range_kernel, dim3((unsigned)ranged, (unsigned)pb.n), 256, 0, st, pb);
      TTNN_TRY(check_launch("tcg_range_kernel"));
    }
    tcg_prepare_kernel<<<(unsigned)blocks, 256, 0, st>>>(pb);
    TTNN_TRY(check_launch("tcg_prepare_kernel"));
  }
  return TTNN_OK;
}

ttnn_status tcg_run(const TcGemm* g, int n, void* pieces, int sms, int* err, uint64_t wait_ns,
                    cudaStream_t st) {
  auto alike = [](const TcGemm& a, const TcGemm& b) {
    return a.type == b.type && a.mn == b.mn && tc::tcg_npad(a) == tc::tcg_npad(b) &&
           tc::tcg_vec(a) == tc::tcg_vec(b);
  };
  std::vector<char> done(n, 0);
  for (int k = 0; k < n; ++k) {
    if (done[k]) continue;
    if (g[k].type == 0) {
      TTNN_TRY(launch_zgemm(g[k], g[k].prep, pieces, sms, err, wait_ns, st));
      continue;
    }
    const TcGemm* batch[kTcgBatch];
    int m = 0;
    int64_t tiles = 0;
    for (int l = k; l < n && m < kTcgBatch; ++l) {
      const int64_t t = ceil_div(g[l].I, (int64_t)tc::kTileM);
      if (done[l] || !alike(g[k], g[l]) || (m > 0 && tiles + t >= (int64_t(1) << 30))) continue;
      batch[m++] = &g[l];
      tiles += t;
      done[l] = 1;
    }
    TTNN_TRY(tc::tcg_batch(batch, m, pieces, sms, err, wait_ns, st));
  }
  return TTNN_OK;
}

ttnn_status launch_tcg(const TcGemm* g, int n, int sms, int* err, uint64_t wait_ns, void* ws,
                       int64_t ws_bytes, cudaStream_t st, bool dry, int64_t* need) {
  int64_t b_bytes = 0, p_bytes = 0;
  std::vector<TcGemm> all(g, g + n), todo;
  std::vector<void*> dst;
  char* w = (char*)ws + (256 - ((uintptr_t)ws & 255)) % 256;
  for (TcGemm& m : all) {
    // the launches run in order and share the room of their pieces
    p_bytes = std::max(p_bytes, tcg_piece_bytes(m, sms));
    if (m.prep) continue;
    todo.push_back(m);
    dst.push_back(w + b_bytes);
    m.prep = w + b_bytes;
    b_bytes += tcg_prep_bytes(m);
  }
  if (dry) {
    *need = b_bytes + p_bytes + 256;
    return TTNN_OK;
  }
  if (w + b_bytes + p_bytes > (char*)ws + ws_bytes) {
    set_error("tensor-core GEMM: workspace too small");
    return TTNN_ENOMEM;
  }
  if (!todo.empty()) TTNN_TRY(tcg_prepare(todo.data(), (int)todo.size(), dst.data(), st));
  return tcg_run(all.data(), n, w + b_bytes, sms, err, wait_ns, st);
}

}  // namespace ttnn
