// Binary64 GEMM on the 16-bit tensor cores (tcgen05), for first-level
// products of binary64 tensors.  The FP64 units of this part run about two
// multiply-adds per clock and SM (1.25 TFLOP/s), so the SIMT GEMM of a 20^6
// tensor took 5.75 ms of a 6.03 ms update; the error-free splitting of Ozaki,
// Ogita, Oishi and Rump (2012) moves the products to the tensor cores.
//
// Every element is a 62-bit integer v at the scale of the largest exponent E
// of its row of A (of its column of B^T): x = v 2^(E - 1084), |v| < 2^62, cut
// towards zero.  v = sum_i d_i 256^(7-i) with eight signed digits |d_i| <= 128,
// each exact in binary16.  Products of digits with i + j = o <= 7 are added
// in one accumulator per order o: over a tile of 32 k that is at most
// 8 * 32 * 2^14 = 2^22, so the binary32 accumulators hold exact integers and
// the tensor core's rounding never acts.  The epilogue adds them to 64-bit
// integers per output (orders 0-3 and 4-7 apart), which are converted and joined
// at the end of a row tile (three roundings where a half has more than 53 bits
// or the result is subnormal, else one); the pieces of a tile that several CTAs
// worked on are added in binary64.
//
// What is left out, orders 8 and up and the cut bits, is below 2^-57 (2^-60 rms)
// of max|a| max|b| per product: an entry far below the largest of its row is held
// in fewer than 53 bits.  In norm the sketches err no more than with multiply-
// adds (eight sizes up to 20^6: 0.84 to 1.02 of it); an entry whose sum of
// |a||b| is far below max|a| max|b|, as in a row of few non-zeros or with one
// outlier, errs more (error over sum |a||b|: Gaussian 6e-17 against 1.1e-16,
// 0.2 % non-zeros 3.5e-15 against 2.6e-16, 20 outliers of 1e10 1.3e-14 against
// 1.5e-15).  TTNN_FLAG_SIMT_PASS keeps the FP64 units.  (With seven digits a 20^6 sketch took 5 % less
// time and erred more than the FP64 units' sums: the columns of B are
// Khatri-Rao products whose largest entry is 100 times their mean.)  Row
// exponents only grow within a sum; when one does, its accumulators are
// shifted.  Digits hold no infinity or NaN: the results of a row (column) with
// one are taken from the operands themselves (zpieces_kernel).
//
// The digits of A are formed by integer instructions in converter warps on
// the way from global to shared memory (no FP64 instruction is used per
// element).  Warp roles (576 threads): warp 0 copies B tiles by TMA, warp 1
// owns TMEM and issues MMAs, warps 2-9 drain accumulators (TMEM lane quarter =
// warp % 4, a half of the columns each), warps 10-17 convert.  Waits are
// bounded as in the other tensor-core kernels.
#include <algorithm>

#include "gemm_tc.cuh"
#include "tc_ptx.cuh"

namespace ttnn {
namespace tc {

constexpr int kZDigits = 8;
constexpr int kZThreads = 576;
constexpr int kZConv = 8;          // converter warps
constexpr int kZK = 32;            // k of an A tile
constexpr int kZBox = 64;          // k of a B tile (two A tiles)
constexpr int kZMaxN = 32;         // columns of one launch
constexpr int kZRing = 8;          // published exponent slots (stages + 2 at least)
constexpr uint32_t kZStage = 65536;   // bytes of an A stage
constexpr int kZBBufs = 2;
constexpr int kZSmem = 1024 + 2 * (int)kZStage + kZBBufs * kZDigits * kZMaxN * 128;   // most a launch takes

struct ZParams {
  const double* A;
  int64_t lda, I, K;
  const double* B;       // [Jn][ldb], the columns of B^T as given
  int64_t ldb;
  int nI, nkb;           // row tiles, B tiles along k
  int Npad, Jn;          // columns of this launch, padded and valid
  int stages;
  const uint32_t* eb;    // [Jn] exponents of the columns of B^T
  double* C;             // [I][ldc], first column of this launch
  int64_t ldc;
  double* part;          // pieces [2 grid][128][Npad]
  int* err;
  uint64_t wait_ns;
};

// The digits of |x| at exponent E: byte 7 - i of the result holds d_i + 128.
__device__ __forceinline__ uint2 digits(uint32_t hi, uint32_t lo, uint32_t E) {
  const uint32_t f = (hi >> 20) & 0x7FFu;
  // the significand with its leading bit at bit 63, moved down to bit 61 and
  // by the distance of the exponents
  const uint32_t mh = (__funnelshift_l(lo, hi, 11) & 0x7FFFFFFFu) | (f ? 0x80000000u : 0u);
  const uint32_t ml = lo << 11;
  const uint32_t sh = E + 2u - (f ? f : 1u);
  uint32_t vh, far;
  asm("shr.u32 %0, %1, %2;" : "=r"(vh) : "r"(mh), "r"(sh));            // 0 from 32 on
  asm("shr.u32 %0, %1, %2;" : "=r"(far) : "r"(mh), "r"(sh - 32u));     // (sh < 32: not used)
  const uint32_t vl = sh < 32u ? __funnelshift_r(ml, mh, sh) : far;
  const uint64_t w = (((uint64_t)vh << 32) | vl) + 0x8080808080808080ull;
  return make_uint2((uint32_t)w, (uint32_t)(w >> 32));
}

// The signs of two elements as binary16 factors +-1 and offsets -+1152.
__device__ __forceinline__ uint2 sign_pair(uint32_t xhi, uint32_t yhi) {
  const uint32_t sg = (__byte_perm(xhi, yhi, 0x7632) & 0x80008000u);
  return make_uint2(0x3C003C00u | sg, 0xE480E480u ^ sg);
}

// binary16 pair of digit I of two elements (x in the low half).
template <int I>
__device__ __forceinline__ uint32_t digit_pair(uint2 x, uint2 y, uint2 sg) {
  constexpr int b = kZDigits - 1 - I;                   // byte of the value
  constexpr uint32_t sel = (uint32_t)(b & 3) | (uint32_t)(4 + (b & 3)) << 8;
  // 1024 + byte, exact in binary16; then +-(1024 + byte) -+ 1152 = +-(byte - 128)
  const uint32_t t = (__byte_perm(b < 4 ? x.x : x.y, b < 4 ? y.x : y.y, sel) & 0x00FF00FFu) | 0x64006400u;
  uint32_t r;
  asm("fma.rn.f16x2 %0, %1, %2, %3;" : "=r"(r) : "r"(t), "r"(sg.x), "r"(sg.y));
  return r;
}

// Larger of the two 16-bit halves each.
__device__ __forceinline__ uint32_t max16x2(uint32_t a, uint32_t b) { return __vmaxu2(a, b); }

// acc + a * b
__device__ __forceinline__ uint64_t mad_wide(uint32_t a, uint32_t b, uint64_t acc) {
  uint64_t r;
  asm("mad.wide.u32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(acc));
  return r;
}

__device__ __forceinline__ void zst(uint32_t addr, uint32_t v) {
  asm volatile("st.shared.b32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}

// Stores digits I..7 of a pair; dst(I) is the address of digit I.
template <int I, typename Dst>
__device__ __forceinline__ void store_digits(uint2 x, uint2 y, uint2 sg, const Dst& dst) {
  if constexpr (I < kZDigits) {
    zst(dst(I), digit_pair<I>(x, y, sg));
    store_digits<I + 1>(x, y, sg, dst);
  }
}

__device__ __forceinline__ void z_tmem_ld8(uint32_t taddr, uint32_t* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7])
      : "r"(taddr));
}

template <bool MN, bool VEC>
__global__ void __launch_bounds__(kZThreads, 1)
    zgemm_kernel(const __grid_constant__ CUtensorMap mapB, const ZParams p) {
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t bar_a[3], bar_empty[3], bar_b[kZBBufs], bar_bfree[kZBBufs];
  __shared__ __align__(8) uint64_t bar_full[2], bar_free[2], bar_done;
  __shared__ uint32_t pub[kZRing][kTileM];   // row exponents of the tile in the slot
  __shared__ uint32_t colmax[4][kTileM];     // MN: column exponents being found
  __shared__ uint32_t tmem_slot;
  __shared__ volatile int abort_flag;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  const uint32_t base = smem_u32(smem);
  const int S = p.stages;
  const uint32_t b_bytes = (uint32_t)(kZDigits * p.Npad * 128);
  const uint32_t b_base = base + S * kZStage;
  // even ranges of the (row tile, B tile) grid, as in the binary32 kernel
  const int64_t total = (int64_t)p.nI * p.nkb;
  const int64_t u0 = total * blockIdx.x / gridDim.x, u1 = total * (blockIdx.x + 1) / gridDim.x;
  const int i0 = (int)(u0 / p.nkb), i1 = u1 > u0 ? (int)((u1 - 1) / p.nkb) + 1 : i0;
  auto range = [&](int it, int* k0, int* k1) {   // B tiles of row tile `it`
    const int64_t r = (int64_t)it * p.nkb;
    *k0 = (int)(max(u0, r) - r);
    *k1 = (int)(min(u1, r + p.nkb) - r);
  };

  if (threadIdx.x == 0) {
    abort_flag = 0;
    for (int s = 0; s < 3; ++s) {
      mbar_init(smem_u32(&bar_a[s]), kZConv);
      mbar_init(smem_u32(&bar_empty[s]), 1);
    }
    for (int s = 0; s < kZBBufs; ++s) {
      mbar_init(smem_u32(&bar_b[s]), 1);
      mbar_init(smem_u32(&bar_bfree[s]), 1);
    }
    for (int k = 0; k < 2; ++k) {
      mbar_init(smem_u32(&bar_full[k]), 1);
      mbar_init(smem_u32(&bar_free[k]), 8);
    }
    mbar_init(smem_u32(&bar_done), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  for (int e = threadIdx.x; e < 4 * kTileM; e += kZThreads) colmax[e / kTileM][e % kTileM] = 0u;
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
  const int acc_cols = kZDigits * p.Npad;   // of one accumulator buffer (at most 256)

  if (warp == 0) {
    if (lane == 0) {
      // ---------------- B tiles by TMA ----------------
      uint64_t pol_keep;
      asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(pol_keep));
      int buf = 0;
      uint32_t ph = 0, used = 0, last_ph = 0;
      bool ok = true;
      for (int it = i0; it < i1 && ok; ++it) {
        int k0, k1;
        range(it, &k0, &k1);
        for (int kb = k0; kb < k1; ++kb) {
          ok = mbar_wait(smem_u32(&bar_bfree[buf]), ph ^ 1, &abort_flag, p.wait_ns);
          if (!ok) break;
          mbar_expect_tx(smem_u32(&bar_b[buf]), b_bytes);
          tma_2d(b_base + buf * b_bytes, &mapB, kb * kZBox, 0, smem_u32(&bar_b[buf]), pol_keep);
          used |= 1u << buf;
          last_ph = (last_ph & ~(1u << buf)) | (ph << buf);
          if (++buf == kZBBufs) {
            buf = 0;
            ph ^= 1;
          }
        }
      }
      if (!ok) {
        abort_flag = 1;
        atomicOr(p.err, 1);
      }
      for (int s = 0; s < kZBBufs; ++s)
        if (((used >> s) & 1u) && !mbar_drain(smem_u32(&bar_b[s]), (last_ph >> s) & 1u))
          atomicOr(p.err, 2);
    }
  } else if (warp == 1) {
    if (lane == 0) {
      // ---------------- MMA issuer ----------------
      int stage = 0, buf = 0, bb = 0;
      uint32_t ph = 0, fph = 1, bph = 0;
      bool ok = true;
      for (int it = i0; it < i1 && ok; ++it) {
        int k0, k1;
        range(it, &k0, &k1);
        for (int kb = k0; kb < k1 && ok; ++kb) {
          ok = mbar_wait(smem_u32(&bar_b[bb]), bph, &abort_flag, p.wait_ns);
          for (int h = 0; h < kZBox / kZK && ok; ++h) {
            ok = mbar_wait(smem_u32(&bar_free[buf]), fph, &abort_flag, p.wait_ns) &&
                 mbar_wait(smem_u32(&bar_a[stage]), ph, &abort_flag, p.wait_ns);
            if (!ok) break;
            fence_after();
            const uint32_t sa = base + stage * kZStage;
            const uint32_t sb = b_base + bb * b_bytes + h * (kZK * 2);
            const uint32_t d = tmem + buf * acc_cols;
            const uint64_t a = sdesc(sa, MN ? 4096 : 16, 1024), b = sdesc(sb, 16, 1024);
#pragma unroll
            for (int i = 0; i < kZDigits; ++i) {
              // digit i of A against digits 0 .. 7 - i of B: orders i .. 7
              const uint32_t id = idesc_f16(kTileM, (kZDigits - i) * p.Npad, MN);
#pragma unroll
              for (int kk = 0; kk < kZK / 16; ++kk) {
                mma_bf16(d + i * p.Npad,
                         sdesc_at(a, MN ? i * 8192 + kk * 2048 : (i >> 1) * 16384 + (i & 1) * 64 + kk * 32),
                         sdesc_at(b, kk * 32), id, i > 0 || kk > 0);
              }
            }
            mma_commit(smem_u32(&bar_empty[stage]));
            mma_commit(smem_u32(&bar_full[buf]));
            if (++stage == S) {
              stage = 0;
              ph ^= 1;
            }
            buf ^= 1;
            if (buf == 0) fph ^= 1;
          }
          if (!ok) break;
          mma_commit(smem_u32(&bar_bfree[bb]));
          if (++bb == kZBBufs) {
            bb = 0;
            bph ^= 1;
          }
        }
      }
      if (!ok) {
        abort_flag = 1;
        atomicOr(p.err, 4);
      }
      mma_commit(smem_u32(&bar_done));
    }
  } else if (warp >= 10) {
    // ---------------- converters ----------------
    const int cw = warp - 10;
    const int64_t rows = MN ? p.K : p.I, cols = MN ? p.I : p.K;
    // pair q of a lane: K-major, row 16 cw + (q & 3) + 8 (q >> 2) + 4 (lane >> 4)
    // and columns 2 (lane & 15), + 1 (rows four apart meet different banks);
    // MN-major, row 4 cw + (q >> 1) and columns 64 (q & 1) + 2 lane, + 1
    constexpr int NP = 8;
    const int rl = MN ? cw * 4 : cw * 16 + 4 * (lane >> 4);
    const int cl = MN ? 2 * lane : 2 * (lane & 15);
    auto row_of = [](int q) { return MN ? q >> 1 : (q & 3) + 8 * (q >> 2); };
    auto col_of = [](int q) { return MN ? 64 * (q & 1) : 0; };
    double2 v[NP];
    int it = i0, kt = 0, kt1 = 0, n = 0;      // A tiles
    const double* src = nullptr;
    int nrow = 0, ncol = 0;
    auto aim = [&]() {
      const int64_t r0 = (MN ? kt * (int64_t)kZK : it * (int64_t)kTileM) + rl;
      const int64_t c0 = (MN ? it * (int64_t)kTileM : kt * (int64_t)kZK) + cl;
      src = p.A + r0 * p.lda + c0;
      nrow = (int)max((int64_t)0, min((int64_t)kTileM, rows - r0));
      ncol = (int)max((int64_t)0, min((int64_t)kTileM, cols - c0));
    };
    auto load = [&](int q) {
      const double* a = src + (int64_t)row_of(q) * p.lda + col_of(q);
      const bool in = row_of(q) < nrow;
      if (VEC) {
        v[q] = in && col_of(q) < ncol ? __ldg(reinterpret_cast<const double2*>(a)) : make_double2(0., 0.);
      } else {
        v[q].x = in && col_of(q) < ncol ? __ldg(a) : 0.;
        v[q].y = in && col_of(q) + 1 < ncol ? __ldg(a + 1) : 0.;
      }
    };
    auto tiles = [&]() {
      int k0, k1;
      range(it, &k0, &k1);
      kt = k0 * (kZBox / kZK);
      kt1 = k1 * (kZBox / kZK);
    };
    if (it < i1) {
      tiles();
      aim();
#pragma unroll
      for (int q = 0; q < NP; ++q) load(q);
    }
    constexpr int NE = MN ? 4 : NP;           // exponents a lane keeps
    uint32_t E[NE];
#pragma unroll
    for (int q = 0; q < NE; ++q) E[q] = 1u;
    int stage = 0;
    uint32_t ph = 0;
    bool ok = true;
    while (it < i1) {
      // exponents of this tile's rows (MN: columns)
      if (!MN) {
#pragma unroll
        for (int q = 0; q < NP; q += 2) {
          // the upper halves of two rows' elements, largest of each row over
          // its 16 lanes (sign cleared: ordered as the exponents are)
          uint32_t e = max16x2(__byte_perm(__double2hiint(v[q].x), __double2hiint(v[q + 1].x), 0x7632) & 0x7FFF7FFFu,
                               __byte_perm(__double2hiint(v[q].y), __double2hiint(v[q + 1].y), 0x7632) & 0x7FFF7FFFu);
#pragma unroll
          for (int o = 8; o > 0; o >>= 1) e = max16x2(e, __shfl_xor_sync(0xffffffffu, e, o));
          E[q] = max(E[q], (e >> 4) & 0x7FFu);
          E[q + 1] = max(E[q + 1], e >> 20);
          if ((lane & 15) == 0) {
            pub[n & (kZRing - 1)][rl + row_of(q)] = E[q];
            pub[n & (kZRing - 1)][rl + row_of(q + 1)] = E[q + 1];
          }
        }
      } else {
#pragma unroll
        for (int c = 0; c < 4; ++c) {         // columns cl + (c & 1) + 64 (c >> 1)
          uint32_t e = 0u;
#pragma unroll
          for (int r = 0; r < 4; ++r) {
            const double x = (c & 1) ? v[2 * r + (c >> 1)].y : v[2 * r + (c >> 1)].x;
            e = max(e, ((uint32_t)__double2hiint(x) >> 20) & 0x7FFu);
          }
          atomicMax(&colmax[n & 3][cl + (c & 1) + 64 * (c >> 1)], e);
        }
        asm volatile("bar.sync 1, %0;" ::"n"(kZConv * 32) : "memory");
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const int col = cl + (c & 1) + 64 * (c >> 1);
          E[c] = max(E[c], colmax[n & 3][col]);
          if (cw == 0) {
            pub[n & (kZRing - 1)][col] = E[c];
            // read by everyone before the barrier of tile n - 1; next used two tiles on
            colmax[(n + 2) & 3][col] = 0u;
          }
        }
      }
      const int it0 = it;
      if (++kt == kt1) {
        ++it;
        if (it < i1) tiles();
      }
      if (it < i1) aim();
      else nrow = 0;
      ok = mbar_wait(smem_u32(&bar_empty[stage]), ph ^ 1, &abort_flag, p.wait_ns);
      if (MN) {
        // the column barrier needs every converter: they stop together
        uint32_t all;
        asm volatile(
            "{\n\t.reg .pred a, b;\n\t"
            "setp.ne.u32 a, %1, 0;\n\t"
            "bar.red.and.pred b, 2, %2, a;\n\t"
            "selp.u32 %0, 1, 0, b;\n\t}\n"
            : "=r"(all)
            : "r"((uint32_t)ok), "n"(kZConv * 32)
            : "memory");
        ok = all != 0u;
      } else {
        ok = __all_sync(0xffffffffu, ok);
      }
      if (!ok) break;
      const uint32_t dst = base + stage * kZStage;
#pragma unroll
      for (int q = 0; q < NP; ++q) {
        const uint32_t ex = MN ? E[MN ? 2 * (q & 1) : 0] : E[MN ? 0 : q];
        const uint32_t ey = MN ? E[MN ? 2 * (q & 1) + 1 : 0] : E[MN ? 0 : q];
        const uint2 x = digits((uint32_t)__double2hiint(v[q].x), (uint32_t)__double2loint(v[q].x), ex);
        const uint2 y = digits((uint32_t)__double2hiint(v[q].y), (uint32_t)__double2loint(v[q].y), ey);
        const uint2 sg = sign_pair((uint32_t)__double2hiint(v[q].x), (uint32_t)__double2hiint(v[q].y));
        const int row = rl + row_of(q);
        if (MN) {
          const uint32_t o = dst + (uint32_t)((q & 1) * 4096 + row * 128) +
                             ((uint32_t)(((lane >> 2) ^ (row & 7)) << 4) + (lane & 3) * 4);
          store_digits<0>(x, y, sg, [&](int i) { return o + i * 8192; });
        } else {
          const uint32_t o = dst + (uint32_t)(row * 128 + (lane & 3) * 4);
          const uint32_t c = (uint32_t)((lane & 15) >> 2), r7 = (uint32_t)(row & 7);
          const uint32_t o0 = o + ((c ^ r7) << 4), o1 = o + (((c + 4) ^ r7) << 4);
          store_digits<0>(x, y, sg, [&](int i) { return (i & 1 ? o1 : o0) + (i >> 1) * 16384; });
        }
        load(q);
      }
      if (it != it0) {
#pragma unroll
        for (int q = 0; q < NE; ++q) E[q] = 1u;
      }
      ++n;
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&bar_a[stage]));
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
    // ---------------- epilogue (warps 2..9) ----------------
    const int q = warp & 3, half = (warp - 2) >> 2;
    const int r_in = 32 * q + lane;
    const int cn = p.Npad / 2, cb = half * cn;   // this warp's columns: 8 or 16
    const uint32_t lane_off = (uint32_t)(32 * q) << 16;
    // bits of a + 1.5 2^23 as an integer are kBias + a: every drain adds the
    // bias of its orders once
    constexpr uint64_t kBias = 0x4B400000ull;
    constexpr uint64_t kBiases = kBias * ((1ull << 24) + (1ull << 16) + (1ull << 8) + 1ull);
    int buf = 0, n = 0;
    uint32_t fph = 0;
    bool ok = true;
    for (int it = i0; it < i1 && ok; ++it) {
      int k0, k1;
      range(it, &k0, &k1);
      uint64_t hi[16], lo[16];
#pragma unroll
      for (int c = 0; c < 16; ++c) hi[c] = lo[c] = 0ull;
      uint32_t E = 0u;
      uint64_t drains = 0;
      for (int t = 0; t < (k1 - k0) * (kZBox / kZK); ++t, ++n) {
        ok = mbar_wait(smem_u32(&bar_full[buf]), fph, &abort_flag, p.wait_ns);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        fence_after();
        const uint32_t e = pub[n & (kZRing - 1)][r_in];
        if (e != E) {
          // the row's exponent grew: its sums so far move down
          const uint32_t dn = min(e - E, 100u);
          if (t > 0) {
#pragma unroll
            for (int c = 0; c < 16; ++c) {
              __int128 T = ((__int128)(int64_t)(hi[c] - drains * kBiases) << 32) +
                           (int64_t)(lo[c] - drains * kBiases);
              T >>= dn;
              hi[c] = (uint64_t)(int64_t)(T >> 32) + drains * kBiases;
              lo[c] = (uint64_t)((int64_t)T & 0xFFFFFFFF) + drains * kBiases;
            }
          }
          E = e;
        }
        const uint32_t d = tmem + lane_off + buf * acc_cols + cb;
#pragma unroll
        for (int g = 0; g < 2; ++g) {
          if (g * 8 >= cn) continue;
          uint32_t a[kZDigits][8];
#pragma unroll
          for (int o = 0; o < kZDigits; ++o) z_tmem_ld8(d + o * p.Npad + g * 8, a[o]);
          tmem_wait_ld();
#pragma unroll
          for (int c = 0; c < 8; ++c) {
            auto bits = [&](int o) { return __float_as_uint(__uint_as_float(a[o][c]) + 12582912.f); };
            uint64_t h = hi[g * 8 + c], l = lo[g * 8 + c];
            h = mad_wide(bits(0), 1u << 24, h);
            h = mad_wide(bits(1), 1u << 16, h);
            h = mad_wide(bits(2), 1u << 8, h);
            h = mad_wide(bits(3), 1u, h);
            l = mad_wide(bits(4), 1u << 24, l);
            l = mad_wide(bits(5), 1u << 16, l);
            l = mad_wide(bits(6), 1u << 8, l);
            l = mad_wide(bits(7), 1u, l);
            hi[g * 8 + c] = h;
            lo[g * 8 + c] = l;
          }
        }
        ++drains;
        fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&bar_free[buf]));
        buf ^= 1;
        if (buf == 0) fph ^= 1;
      }
      if (!ok) break;
      const bool whole = k0 == 0 && k1 == p.nkb;
      const int64_t row = (int64_t)it * kTileM + r_in;
      if (row < p.I) {
        double* out = whole ? p.C + row * p.ldc + cb
                            : p.part + ((int64_t)(2 * blockIdx.x + (it > i0)) * kTileM + r_in) * p.Npad + cb;
#pragma unroll
        for (int c = 0; c < 16; ++c) {
          if (c >= cn) continue;
          const uint32_t eb = cb + c < p.Jn ? __ldg(p.eb + cb + c) : 1u;
          const double T = __fma_rn((double)(int64_t)(hi[c] - drains * kBiases), 4294967296.0,
                                    (double)(int64_t)(lo[c] - drains * kBiases));
          const double r = scalbn(T, (int)E + (int)eb - 2112);
          out[c] = E == 0x7FFu || eb == 0x7FFu ? __longlong_as_double(0x7FF8000000000000ll) : r;
        }
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

// A prepared operand: the exponents of its columns (1024 bytes), then the
// digits as the kernel's TMA reads them, per column group of kZMaxN:
// [8][Npad][Kpad] binary16, zero beyond the operand.
constexpr int kZExpBytes = 1024;
struct ZPrepJob {
  const double* B;
  uint32_t* eb;
  uint32_t* out;
  int64_t ldb, K, Kpad;
  int Jn, W;
};
struct ZPrepBatch {
  ZPrepJob job[2];
};

// Largest exponent field of every row of B (eb zeroed before).
__global__ void __launch_bounds__(256) zmax_kernel(const __grid_constant__ ZPrepBatch b) {
  const ZPrepJob& j = b.job[blockIdx.z];
  const int r = blockIdx.y;
  if (r >= j.Jn) return;
  const double* row = j.B + r * j.ldb;
  uint32_t e = 1u;
  for (int64_t k = blockIdx.x * 256ll + threadIdx.x; k < j.K; k += (int64_t)gridDim.x * 256)
    e = max(e, ((uint32_t)__double2hiint(row[k]) >> 20) & 0x7FFu);
  e = __reduce_max_sync(0xffffffffu, e);
  if ((threadIdx.x & 31) == 0) atomicMax(j.eb + r, e);
}

__global__ void __launch_bounds__(256) zslice_kernel(const __grid_constant__ ZPrepBatch b) {
  const ZPrepJob& j = b.job[blockIdx.z];
  const int r = blockIdx.y;                               // column of the product, padded
  if (r >= j.W) return;
  const int64_t half = j.Kpad / 2;
  const int g0 = r / kZMaxN * kZMaxN;
  const int Npad = min(kZMaxN, j.W - g0);
  uint32_t* o = j.out + (int64_t)g0 * kZDigits * half + (int64_t)(r - g0) * half;
  const uint32_t E = r < j.Jn ? j.eb[r] : 1u;
  for (int64_t e = blockIdx.x * 256ll + threadIdx.x; e < half; e += (int64_t)gridDim.x * 256) {
    const int64_t k = 2 * e;
    const double x = r < j.Jn && k < j.K ? j.B[r * j.ldb + k] : 0.;
    const double y = r < j.Jn && k + 1 < j.K ? j.B[r * j.ldb + k + 1] : 0.;
    const uint2 dx = digits((uint32_t)__double2hiint(x), (uint32_t)__double2loint(x), E);
    const uint2 dy = digits((uint32_t)__double2hiint(y), (uint32_t)__double2loint(y), E);
    const uint2 sg = sign_pair((uint32_t)__double2hiint(x), (uint32_t)__double2hiint(y));
    auto put = [&](int i, uint32_t w) { o[(int64_t)i * Npad * half + e] = w; };
    put(0, digit_pair<0>(dx, dy, sg));
    put(1, digit_pair<1>(dx, dy, sg));
    put(2, digit_pair<2>(dx, dy, sg));
    put(3, digit_pair<3>(dx, dy, sg));
    put(4, digit_pair<4>(dx, dy, sg));
    put(5, digit_pair<5>(dx, dy, sg));
    put(6, digit_pair<6>(dx, dy, sg));
    put(7, digit_pair<7>(dx, dy, sg));
  }
}

// C(row, col) from the operands, in order, up to the first NaN.
template <bool MN>
__device__ __noinline__ double z_direct(const ZParams& p, int64_t row, int col) {
  const double* x = p.A + row * (MN ? 1 : p.lda);
  const double* y = p.B + col * p.ldb;
  double a = 0.;
  for (int64_t k = 0; k < p.K && !isnan(a); ++k) a = __fma_rn(x[k * (MN ? p.lda : 1)], y[k], a);
  return a;
}

// Sums the pieces of the row tiles that more than one CTA worked on.  Where an
// infinity or NaN of A or B has left NaN, the entry is summed from the operands
// by multiply-adds, as the FP64 units would (up to the first NaN of its sum).
// Whole tiles are looked over for that as well: a read of C.
template <bool MN>
__global__ void __launch_bounds__(256) zpieces_kernel(const __grid_constant__ ZParams p, int G) {
  const int it = blockIdx.x, nkb = p.nkb, Npad = p.Npad;
  const int64_t total = (int64_t)p.nI * nkb;
  auto owner = [&](int64_t u) { return (int)(((u + 1) * G - 1) / total); };
  const int c0 = owner((int64_t)it * nkb), c1 = owner((int64_t)(it + 1) * nkb - 1);
  const int rows = (int)min((int64_t)kTileM, p.I - (int64_t)it * kTileM);
  const int64_t tile = (int64_t)kTileM * Npad;
  // only the first CTA's range can begin in an earlier tile
  const double* p0 = p.part + (int64_t)(2 * c0 + ((int)(total * c0 / G / nkb) < it)) * tile;
  for (int e = blockIdx.y * 256 + threadIdx.x; e < rows * Npad; e += gridDim.y * 256) {
    const int64_t row = (int64_t)it * kTileM + e / Npad;
    const int col = e % Npad;
    double* out = p.C + row * p.ldc + col;
    double a = c0 == c1 ? *out : p0[e];
#pragma unroll 4
    for (int c = c0 + 1; c <= c1; ++c) a += p.part[(int64_t)(2 * c) * tile + e];
    const bool redo = ((uint32_t)__double2hiint(a) & 0x7FFFFFFFu) > 0x7FF00000u && col < p.Jn;   // a NaN
    if (redo) a = z_direct<MN>(p, row, col);
    if (redo || c0 != c1) *out = a;
  }
}

struct ZGeometry {
  int W, nI, nkb, stages, grid;     // W: padded columns of all groups
  int64_t Kpad, b_bytes, p_bytes;
  size_t smem;
};

static ZGeometry z_geometry(const TcGemm& g, int sms) {
  ZGeometry o;
  o.W = (int)round_up(g.Jn, 16);
  o.nI = (int)ceil_div(g.I, (int64_t)kTileM);
  o.nkb = (int)ceil_div(g.K, (int64_t)kZBox);
  o.Kpad = (int64_t)o.nkb * kZBox;
  const int N = std::min(o.W, kZMaxN);
  o.stages = 2;
  o.smem = (size_t)(1024 + o.stages * kZStage + kZBBufs * kZDigits * N * 128);
  o.grid = (int)std::max<int64_t>(1, std::min<int64_t>((int64_t)o.nI * o.nkb, sms));
  o.b_bytes = round_up((int64_t)kZDigits * o.W * o.Kpad * 2, 256) + kZExpBytes;
  o.p_bytes = (int64_t)2 * sms * kTileM * N * 8;
  return o;
}

template <bool MN, bool VEC>
static ttnn_status z_launch(const ZGeometry& o, const CUtensorMap& mB, const ZParams& p, cudaStream_t st) {
  constexpr int slot = 32 + (MN ? 2 : 0) + (VEC ? 1 : 0);
  TTNN_TRY(smem_limit_once((const void*)zgemm_kernel<MN, VEC>, slot, kZSmem));
  zgemm_kernel<MN, VEC><<<o.grid, kZThreads, o.smem, st>>>(mB, p);
  return check_launch("zgemm_kernel");
}

}  // namespace tc

bool zgemm_supported(const TcGemm& g) {
  const int64_t lim = int64_t(1) << 31;
  if (g.type != 0 || g.I < 1 || g.Jn < 1 || g.K < 1 || g.Jn > 256) return false;
  if (g.trans || g.nb != 1 || g.b[0].nkr || g.b[0].sk != 1) return false;
  // 64-bit integer sums of 2^46 per drain of 32 k; 32-bit tile counts
  return g.K <= (int64_t(1) << 21) && g.I < lim - 256 && g.ldc == round_up(g.Jn, 16);
}

int64_t zgemm_prep_bytes(const TcGemm& g) { return tc::z_geometry(g, 1).b_bytes; }
int64_t zgemm_piece_bytes(const TcGemm& g, int sms) { return tc::z_geometry(g, sms).p_bytes; }

ttnn_status zgemm_prepare(const TcGemm* g, int n, void* const* dst, cudaStream_t st) {
  using namespace tc;
  ZPrepBatch b;
  int64_t most = 1;
  int w = 0;
  for (int k = 0; k < n; ++k) {
    const ZGeometry o = z_geometry(g[k], 1);
    ZPrepJob& j = b.job[k];
    j.B = (const double*)g[k].b[0].p;
    j.eb = (uint32_t*)dst[k];
    j.out = (uint32_t*)((char*)dst[k] + kZExpBytes);
    j.ldb = g[k].b[0].sj;
    j.K = g[k].K;
    j.Kpad = o.Kpad;
    j.Jn = g[k].Jn;
    j.W = o.W;
    most = std::max(most, g[k].K);
    w = std::max(w, o.W);
    TTNN_TRY_CUDA(cudaMemsetAsync(dst[k], 0, kZExpBytes, st));
  }
  const dim3 grid((unsigned)std::min<int64_t>(ceil_div(most, (int64_t)1024), 64), (unsigned)w, (unsigned)n);
  zmax_kernel<<<grid, 256, 0, st>>>(b);
  TTNN_TRY(check_launch("zmax_kernel"));
  zslice_kernel<<<grid, 256, 0, st>>>(b);
  return check_launch("zslice_kernel");
}

ttnn_status launch_zgemm(const TcGemm& g, const void* prep, void* pieces, int sms, int* err,
                         uint64_t wait_ns, cudaStream_t st) {
  using namespace tc;
  const ZGeometry o = z_geometry(g, sms);
  const uint16_t* dig = (const uint16_t*)((const char*)prep + kZExpBytes);
  for (int j0 = 0; j0 < o.W; j0 += kZMaxN) {
    ZParams p;
    p.A = (const double*)g.A;
    p.lda = g.lda;
    p.I = g.I;
    p.K = g.K;
    p.B = (const double*)g.b[0].p + j0 * g.b[0].sj;
    p.ldb = g.b[0].sj;
    p.nI = o.nI;
    p.nkb = o.nkb;
    p.Npad = std::min(kZMaxN, o.W - j0);
    p.Jn = (int)std::min<int64_t>(p.Npad, g.Jn - j0);
    p.stages = o.stages;
    p.eb = (const uint32_t*)prep + j0;
    p.C = (double*)g.C + j0;
    p.ldc = g.ldc;
    p.part = (double*)pieces;
    p.err = err;
    p.wait_ns = wait_ns;
    CUtensorMap mB;
    TTNN_TRY(encode_map(&mB, dig + (int64_t)j0 * kZDigits * o.Kpad, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2,
                        o.Kpad, (int64_t)kZDigits * p.Npad, (uint32_t)kZBox,
                        (uint32_t)(kZDigits * p.Npad), CU_TENSOR_MAP_SWIZZLE_128B));
    const int64_t inner = g.mn ? g.I : g.K;
    const bool vec = inner % 2 == 0 && g.lda % 2 == 0 && (uintptr_t)g.A % 16 == 0;
    if (g.mn) TTNN_TRY(vec ? z_launch<true, true>(o, mB, p, st) : z_launch<true, false>(o, mB, p, st));
    else TTNN_TRY(vec ? z_launch<false, true>(o, mB, p, st) : z_launch<false, false>(o, mB, p, st));
    const int per = (int)std::max<int64_t>(1, std::min<int64_t>(16, 2432 / std::max(1, o.nI)));
    const dim3 pg((unsigned)o.nI, (unsigned)per);
    if (g.mn) zpieces_kernel<true><<<pg, 256, 0, st>>>(p, o.grid);
    else zpieces_kernel<false><<<pg, 256, 0, st>>>(p, o.grid);
    TTNN_TRY(check_launch("zpieces_kernel"));
  }
  return TTNN_OK;
}

}  // namespace ttnn
