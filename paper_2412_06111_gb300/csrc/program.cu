// Batched executor of small-contraction programs (see program.cuh).
#include <algorithm>
#include <cstring>
#include <type_traits>

#include <cstdio>

#include "program.cuh"

namespace ttnn {

constexpr int kExecThreads = 256;
static_assert(sizeof(LevelBatch<WalkOp, kLargeOps>) <= 32000 &&
                  sizeof(LevelBatch<CpOp, kLargeOps>) <= 32000,
              "level batch must fit the kernel parameter space");
constexpr int kMpKC2 = 32;
constexpr size_t kExecSmem = 48 * 1024;
constexpr size_t kKgemmSmem = 48 * 1024;
constexpr size_t kLaneSmem = 8 * 32 * 8;   // one partial sum per thread of a block

static int exec_sms() {
  static int n = 0;
  if (!n) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    if (n <= 0) n = 148;
  }
  return n;
}

// ---------------------------------------------------------------------------
// device parts
// ---------------------------------------------------------------------------
template <typename Tin, typename Tw, typename Tout, typename Tacc, typename I>
__device__ void dev_contract(const WalkOp& op, int64_t blk) {
  const Contract& c = op.c;
  const int g = op.g;
  const I J = (I)c.J, Q = (I)c.Q, NB = (I)c.NB;
  const I total = (I)(c.P * c.NB * c.Q * c.J);
  const I vo = (I)(blk * (kExecThreads / g)) + (I)(threadIdx.x / g);
  const int lg = threadIdx.x % g;
  const bool valid = vo < total * (I)op.nsplit;
  Tacc acc = 0;
  I split = 0, o = 0, p = 0, b = 0, q = 0, j = 0;
  if (valid) {
    split = vo / total;
    o = vo - split * total;
    I t = o;
    j = t % J;
    t /= J;
    q = t % Q;
    t /= Q;
    b = t % NB;
    p = t / NB;
    const int64_t i0 = (int64_t)split * op.chunk;
    const int64_t i1 = min(c.NI, i0 + op.chunk);
    const Tin* ip = (const Tin*)c.in + (int64_t)p * c.isP + (int64_t)q * c.isQ + (int64_t)j * c.isJ;
    // four independent partial sums: loads and multiply-adds of different
    // terms overlap instead of waiting on one accumulator
    Tacc a1 = 0, a2 = 0, a3 = 0;
    int64_t i = i0 + lg;
    if (c.w) {
      const Tw* wp = (const Tw*)c.w + (int64_t)p * c.wsP + (int64_t)b * c.wsB + (int64_t)q * c.wsQ +
                     (int64_t)j * c.wsJ;
      for (; i + 3 * g < i1; i += 4 * g) {
        acc += (Tacc)ip[i * c.isI] * (Tacc)wp[i * c.wsI];
        a1 += (Tacc)ip[(i + g) * c.isI] * (Tacc)wp[(i + g) * c.wsI];
        a2 += (Tacc)ip[(i + 2 * g) * c.isI] * (Tacc)wp[(i + 2 * g) * c.wsI];
        a3 += (Tacc)ip[(i + 3 * g) * c.isI] * (Tacc)wp[(i + 3 * g) * c.wsI];
      }
      for (; i < i1; i += g) acc += (Tacc)ip[i * c.isI] * (Tacc)wp[i * c.wsI];
    } else {
      for (; i + 3 * g < i1; i += 4 * g) {
        acc += (Tacc)ip[i * c.isI];
        a1 += (Tacc)ip[(i + g) * c.isI];
        a2 += (Tacc)ip[(i + 2 * g) * c.isI];
        a3 += (Tacc)ip[(i + 3 * g) * c.isI];
      }
      for (; i < i1; i += g) acc += (Tacc)ip[i * c.isI];
    }
    acc = (acc + a1) + (a2 + a3);
  }
  for (int off = g >> 1; off > 0; off >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, off);
  if (valid && lg == 0) {
    if (op.nsplit > 1) {
      ((Tout*)op.partial)[(int64_t)split * total + o] = (Tout)acc;
    } else {
      Tout* out = (Tout*)c.out;
      const int64_t oi = (int64_t)p * c.osP + (int64_t)b * c.osB + (int64_t)q * c.osQ + (int64_t)j * c.osJ;
      const Tout v = (Tout)((Tacc)c.alpha * acc);
      out[oi] = c.accumulate ? (Tout)(out[oi] + v) : v;
    }
  }
}

template <typename T, typename I>
__device__ void dev_reduce(const WalkOp& op, int64_t blk) {
  const Contract& c = op.c;
  const I total = (I)(c.P * c.NB * c.Q * c.J);
  const I o = (I)(blk * kExecThreads) + (I)threadIdx.x;
  if (o >= total) return;
  const T* part = (const T*)op.partial;
  T acc = 0;
  for (int s = 0; s < op.nsplit; ++s) acc += part[(int64_t)s * total + o];
  I t = o;
  const I j = t % (I)c.J;
  t /= (I)c.J;
  const I q = t % (I)c.Q;
  t /= (I)c.Q;
  const I b = t % (I)c.NB;
  const I p = t / (I)c.NB;
  T* out = (T*)c.out;
  const int64_t oi = (int64_t)p * c.osP + (int64_t)b * c.osB + (int64_t)q * c.osQ + (int64_t)j * c.osJ;
  const T v = (T)c.alpha * acc;
  out[oi] = c.accumulate ? out[oi] + v : v;
}

// Contraction with a contiguous axis across the lanes: the columns j (op.CH =
// 0: isJ = 1, weights shared with the column or not) or the outputs b (op.CH =
// 1: J = 1, wsB = 1, every lane reads the same input).  op.BG lanes take an
// item (8, 16 or 32: the least that hold the axis, which is cut beyond 32) and
// op.CG warps of a block share its reduction index, summed in warp order.  A
// lane group per output (OP_CONTRACT) reads one element of each row per lane
// when it cuts the reduction index: 200 x 200 x 30 sums of a TTN update took
// 76 us for 48 MB; rows are read whole here.
template <typename Tin, typename Tw, typename T, typename I>
__device__ void dev_lane(const WalkOp& op, int64_t blk, unsigned char* smem) {
  const Contract& c = op.c;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int LW = op.BG, WS = op.CG;
  const bool jl = op.CH == 0;
  const I LN = (I)(jl ? c.J : c.NB);
  const I nch = (LN + LW - 1) / LW;
  const I NBi = jl ? (I)c.NB : (I)1, Q = (I)c.Q;
  const I items = (I)c.P * NBi * Q, units = items * nch * (I)op.nsplit;
  const int per = 32 / LW;
  const I u = ((I)(blk * (8 / WS)) + (I)(warp / WS)) * per + (I)(lane / LW);
  const int s = warp % WS;
  const bool valid = u < units;
  I l = 0, p = 0, b = 0, q = 0, split = 0;
  T acc = 0;
  if (valid) {
    const I ch = u % nch;
    I t = u / nch;
    l = ch * LW + (I)(lane % LW);
    split = t / items;
    t -= split * items;
    q = t % Q;
    t /= Q;
    b = t % NBi;
    p = t / NBi;
    if (l < LN) {
      const int64_t a0 = (int64_t)split * op.chunk, a1 = min(c.NI, a0 + op.chunk);
      const int64_t part = (a1 - a0 + WS - 1) / WS;
      int64_t i = a0 + s * part;
      const int64_t i1 = min(a1, i + part);
      const Tin* ip = (const Tin*)c.in + (int64_t)p * c.isP + (int64_t)q * c.isQ + (jl ? (int64_t)l * c.isJ : 0);
      T a1s = 0, a2s = 0, a3s = 0;
      if (c.w) {
        const Tw* wp = (const Tw*)c.w + (int64_t)p * c.wsP + (int64_t)q * c.wsQ +
                       (jl ? (int64_t)b * c.wsB + (int64_t)l * c.wsJ : (int64_t)l * c.wsB);
        for (; i + 7 < i1; i += 8) {
          T x[8], y[8];
#pragma unroll
          for (int k = 0; k < 8; ++k) {
            x[k] = (T)ip[(i + k) * c.isI];
            y[k] = (T)wp[(i + k) * c.wsI];
          }
          acc += x[0] * y[0];
          a1s += x[1] * y[1];
          a2s += x[2] * y[2];
          a3s += x[3] * y[3];
          acc += x[4] * y[4];
          a1s += x[5] * y[5];
          a2s += x[6] * y[6];
          a3s += x[7] * y[7];
        }
        for (; i < i1; ++i) acc += (T)ip[i * c.isI] * (T)wp[i * c.wsI];
      } else {
        for (; i + 3 < i1; i += 4) {
          acc += (T)ip[i * c.isI];
          a1s += (T)ip[(i + 1) * c.isI];
          a2s += (T)ip[(i + 2) * c.isI];
          a3s += (T)ip[(i + 3) * c.isI];
        }
        for (; i < i1; ++i) acc += (T)ip[i * c.isI];
      }
      acc = (acc + a1s) + (a2s + a3s);
    }
  }
  if (WS > 1) {
    T* red = (T*)smem;   // [8][32]
    red[warp * 32 + lane] = acc;
    __syncthreads();
    if (s != 0) return;
    for (int k = 1; k < WS; ++k) acc += red[(warp + k) * 32 + lane];
  }
  if (!valid || l >= LN) return;
  const I j = jl ? l : (I)0;
  if (!jl) b = l;
  if (op.nsplit > 1) {
    const int64_t o = (((int64_t)p * c.NB + b) * c.Q + q) * c.J + j;
    ((T*)op.partial)[(int64_t)split * (c.P * c.NB * c.Q * c.J) + o] = acc;
  } else {
    T* out = (T*)c.out + (int64_t)p * c.osP + (int64_t)b * c.osB + (int64_t)q * c.osQ + (int64_t)j * c.osJ;
    const T v = (T)c.alpha * acc;
    *out = c.accumulate ? *out + v : v;
  }
}

// Mode product as a batched small GEMM over one chunk of CH batch items:
// out[p,b,q,j] (+)= alpha * sum_i W[i*wsI + b*wsB] * in[p,i,q,j].
template <typename T, typename I>
__device__ void dev_mp(const WalkOp& op, int64_t blk, unsigned char* smem) {
  const Contract& c = op.c;
  const int BG = op.BG, CG = op.CG, CH = op.CH;
  const int WB = 4 * BG, WC = 4 * CG;
  T* Ws = (T*)smem;                   // [kMpKC2][WB]
  T* Is = Ws + kMpKC2 * WB;           // [kMpKC2][WC]
  const int tid = threadIdx.x;
  const int bg = tid / CG, cg = tid % CG;
  const int J = (int)c.J;
  const int ncol = CH * J;
  const I items = (I)(c.P * c.Q);
  const I Qi = (I)c.Q;
  const I it0 = (I)(blk * CH);
  // fixed load column of this thread (WC divides the block size)
  const int lcol = tid % WC, lrow0 = tid / WC, lstep = kExecThreads / WC;
  bool lvalid = false;
  int64_t lbase = 0;
  if (lcol < ncol) {
    const I item = it0 + (I)(lcol / J);
    if (item < items) {
      const I p = item / Qi, q = item - p * Qi;
      lbase = (int64_t)p * c.isP + (int64_t)q * c.isQ + (int64_t)(lcol % J) * c.isJ;
      lvalid = true;
    }
  }
  const int wcol = tid % WB, wrow0 = tid / WB, wstep = kExecThreads / WB;
  const T* in = (const T*)c.in;
  const T* w = (const T*)c.w;
  T acc[4][4];
#pragma unroll
  for (int x = 0; x < 4; ++x)
#pragma unroll
    for (int y = 0; y < 4; ++y) acc[x][y] = 0;
  for (int64_t i0 = 0; i0 < c.NI; i0 += kMpKC2) {
    const int kc = (int)min((int64_t)kMpKC2, c.NI - i0);
    __syncthreads();
    for (int ii = wrow0; ii < kc; ii += wstep)
      Ws[ii * WB + wcol] = (wcol < c.NB) ? w[(i0 + ii) * c.wsI + wcol * c.wsB] : (T)0;
    for (int ii = lrow0; ii < kc; ii += lstep)
      Is[ii * WC + lcol] = lvalid ? in[lbase + (i0 + ii) * c.isI] : (T)0;
    __syncthreads();
    if (bg < BG) {
      for (int ii = 0; ii < kc; ++ii) {
        // 4 consecutive elements per thread: one vector load each (the column
        // tile is read conflict-free, the weight tile is a broadcast)
        T a[4], bb[4];
        if (sizeof(T) == 4) {
          const float4 av = *reinterpret_cast<const float4*>(&Ws[ii * WB + 4 * bg]);
          const float4 bv = *reinterpret_cast<const float4*>(&Is[ii * WC + 4 * cg]);
          a[0] = (T)av.x; a[1] = (T)av.y; a[2] = (T)av.z; a[3] = (T)av.w;
          bb[0] = (T)bv.x; bb[1] = (T)bv.y; bb[2] = (T)bv.z; bb[3] = (T)bv.w;
        } else {
#pragma unroll
          for (int x = 0; x < 4; ++x) {
            a[x] = Ws[ii * WB + 4 * bg + x];
            bb[x] = Is[ii * WC + 4 * cg + x];
          }
        }
#pragma unroll
        for (int x = 0; x < 4; ++x)
#pragma unroll
          for (int y = 0; y < 4; ++y) acc[x][y] += a[x] * bb[y];
      }
    }
  }
  if (bg >= BG) return;
#pragma unroll
  for (int y = 0; y < 4; ++y) {
    const int col = 4 * cg + y;
    if (col >= ncol) continue;
    const I item = it0 + (I)(col / J);
    if (item >= items) continue;
    const int j = col % J;
    const I p = item / Qi, q = item - p * Qi;
    T* out = (T*)c.out;
#pragma unroll
    for (int x = 0; x < 4; ++x) {
      const int b = 4 * bg + x;
      if (b >= c.NB) continue;
      const int64_t oi = (int64_t)p * c.osP + (int64_t)b * c.osB + (int64_t)q * c.osQ + (int64_t)j * c.osJ;
      const T v = (T)c.alpha * acc[x][y];
      out[oi] = c.accumulate ? out[oi] + v : v;
    }
  }
}

// Mode product, weight-stationary: W (NI x NB, NI <= 128, NB <= NBT) sits
// in shared memory; each thread owns one output column (an (item, j) pair)
// and all NB outputs of it in registers, streaming its NI inputs.
// out[p,b,q,j] (+)= alpha * sum_i W[i*wsI + b*wsB] * in[p,i,q,j].
constexpr int kWsMaxNI = 128;

template <int NBT, typename I>
__device__ void dev_mpw(const WalkOp& op, int64_t blk, unsigned char* smem) {
  const Contract& c = op.c;
  float* Ws = (float*)smem;                 // [NI][NBT]
  const int NI = (int)c.NI, NB = (int)c.NB;
  const float* w = (const float*)c.w;
  for (int e = threadIdx.x; e < NI * NBT; e += kExecThreads) {
    const int i = e / NBT, b = e % NBT;
    Ws[e] = b < NB ? w[(int64_t)i * c.wsI + (int64_t)b * c.wsB] : 0.f;
  }
  __syncthreads();
  const I J = (I)c.J, Q = (I)c.Q;
  const I ncols = (I)(c.P * c.Q * c.J);
  const I col = (I)(blk * kExecThreads) + (I)threadIdx.x;
  if (col >= ncols) return;
  const I item = col / J, j = col - item * J;
  const I p = item / Q, q = item - p * Q;
  const float* in = (const float*)c.in + (int64_t)p * c.isP + (int64_t)q * c.isQ + (int64_t)j * c.isJ;
  float acc[NBT];
#pragma unroll
  for (int b = 0; b < NBT; ++b) acc[b] = 0.f;
  int i = 0;
  for (; i + 4 <= NI; i += 4) {
    float x[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) x[u] = in[(int64_t)(i + u) * c.isI];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const float4* wr = reinterpret_cast<const float4*>(Ws + (i + u) * NBT);
#pragma unroll
      for (int b4 = 0; b4 < NBT / 4; ++b4) {
        const float4 wv = wr[b4];
        acc[4 * b4] += wv.x * x[u];
        acc[4 * b4 + 1] += wv.y * x[u];
        acc[4 * b4 + 2] += wv.z * x[u];
        acc[4 * b4 + 3] += wv.w * x[u];
      }
    }
  }
  for (; i < NI; ++i) {
    const float x = in[(int64_t)i * c.isI];
    const float4* wr = reinterpret_cast<const float4*>(Ws + i * NBT);
#pragma unroll
    for (int b4 = 0; b4 < NBT / 4; ++b4) {
      const float4 wv = wr[b4];
      acc[4 * b4] += wv.x * x;
      acc[4 * b4 + 1] += wv.y * x;
      acc[4 * b4 + 2] += wv.z * x;
      acc[4 * b4 + 3] += wv.w * x;
    }
  }
  float* out = (float*)c.out + (int64_t)p * c.osP + (int64_t)q * c.osQ + (int64_t)j * c.osJ;
  const float alpha = (float)c.alpha;
#pragma unroll
  for (int b = 0; b < NBT; ++b) {
    if (b < NB) {
      float* o = out + (int64_t)b * c.osB;
      *o = c.accumulate ? *o + alpha * acc[b] : alpha * acc[b];
    }
  }
}

// Long reduction of a mode product with few batch items (e.g. Y_t^T G_t over
// all rows of a node): block (item, split) sums its K slice of
// out[p,b,q,j] = sum_i W[i*wsI + b*wsB] in[p,i,q,j] through shared-memory
// tiles (coalesced loads) into partial[split][p][b][q][j].
constexpr int kKredTile = 64;

__device__ void dev_kred(const WalkOp& op, int64_t blk, unsigned char* smem) {
  const Contract& c = op.c;
  const int NB = (int)c.NB, J = (int)c.J;
  const int64_t items = c.P * c.Q;
  const int64_t item = blk % items;
  const int64_t split = blk / items;
  const int64_t p = item / c.Q, q = item % c.Q;
  const int64_t i0 = split * op.chunk;
  const int64_t i1 = min(c.NI, i0 + op.chunk);
  float* Wt = (float*)smem;                    // [kKredTile][NB]
  float* It = Wt + kKredTile * 64;             // [kKredTile][J]
  const float* in = (const float*)c.in + p * c.isP + q * c.isQ;
  const float* w = (const float*)c.w;
  const int nout = NB * J;
  float acc[16];
#pragma unroll
  for (int k = 0; k < 16; ++k) acc[k] = 0.f;
  for (int64_t t0 = i0; t0 < i1; t0 += kKredTile) {
    const int kc = (int)min((int64_t)kKredTile, i1 - t0);
    __syncthreads();
    for (int e = threadIdx.x; e < kKredTile * NB; e += kExecThreads) {
      const int b = e / kKredTile, ii = e % kKredTile;   // consecutive threads: consecutive i
      Wt[ii * 64 + b] = ii < kc ? w[(t0 + ii) * c.wsI + (int64_t)b * c.wsB] : 0.f;
    }
    for (int e = threadIdx.x; e < kKredTile * J; e += kExecThreads) {
      const int ii = e / J, jj = e % J;                 // consecutive threads: consecutive j
      It[ii * J + jj] = ii < kc ? in[(t0 + ii) * c.isI + (int64_t)jj * c.isJ] : 0.f;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 16; ++k) {
      const int o = threadIdx.x + k * kExecThreads;
      if (o < nout) {
        const int b = o / J, jj = o % J;
        float a = acc[k];
        for (int ii = 0; ii < kc; ++ii) a += Wt[ii * 64 + b] * It[ii * J + jj];
        acc[k] = a;
      }
    }
  }
  float* part = (float*)op.partial;
  const int64_t total = c.P * c.NB * c.Q * c.J;
#pragma unroll
  for (int k = 0; k < 16; ++k) {
    const int o = threadIdx.x + k * kExecThreads;
    if (o < nout) {
      const int b = o / J, jj = o % J;
      part[split * total + ((p * c.NB + b) * c.Q + q) * c.J + jj] = acc[k];
    }
  }
}

// Split-K register-tiled contraction for long reductions (e.g. the
// Khatri-Rao contraction of all leading modes of a first-level product at
// once, or a TTN core against a sketch block):
//   out[p,b,q,j] (+)= alpha * sum_i W(i, b) in[p,i,q,j],
// with W(i, b) = w[i*wsI + b*wsB] or the Khatri-Rao product of the factors
// c.kr (nkr > 0).  Columns n = (p, q, j) are tiled kKgNT per block, the
// outputs b in groups of kKgMB (op.BG groups) and the reduction index in
// chunks of op.chunk: block = (tile, b group, split).  Each thread
// accumulates 8 (b) x 4 (n) outputs from shared-memory tiles of kKgKT rows,
// the next rows prefetched into registers.  Tiles are read column-wise
// (consecutive threads, consecutive columns: contiguous j) or, with op.CG = 1
// (J = Q = 1 and a contiguous reduction index), row-wise (16 consecutive i of
// a column per 16 threads).  With nsplit > 1 the block writes its partial
// sums [split][p][b][q][j], reduced in a fixed order (OP_REDUCE), else the
// outputs.
constexpr int kKgKT = 16, kKgNT = 256, kKgMB = 32;
constexpr int kKgLd = kKgNT + 4;               // padded tile row (row-wise stores: 2-way banks)
constexpr int kKgWPT = kKgKT * kKgMB / 256;   // weight-tile entries per thread
static_assert(kKgKT * kKgMB % 256 == 0 && kKgWPT >= 1, "weight tile must split over 256 threads");
static_assert(kKgKT == 16 && kKgNT == 256, "row-wise tile loads assume 16 x 256 tiles");

// W(i, b) of a split-K contraction; i < 2^31 (the recorder checks).
__device__ __forceinline__ float kg_weight(const Contract& c, int64_t i, int b) {
  if (c.nkr == 0) return ((const float*)c.w)[i * c.wsI + (int64_t)b * c.wsB];
  float v = 1.f;
  uint32_t rem = (uint32_t)i;
#pragma unroll
  for (int f = 3; f >= 0; --f) {
    if (f >= c.nkr) continue;
    const uint32_t n = (uint32_t)c.krn[f];
    const uint32_t q = rem / n;
    const uint32_t d = rem - q * n;
    rem = q;
    v *= ((const float*)c.kr[f])[(int64_t)d * c.wsI + (int64_t)b * c.wsB];
  }
  return v;
}

template <typename I>
__device__ void dev_kgemm(const WalkOp& op, int64_t blk, unsigned char* smem) {
  const Contract& c = op.c;
  float* Ws = (float*)smem;                       // [kKgKT][kKgMB]
  float* Is = Ws + kKgKT * kKgMB;                 // [kKgKT][kKgLd]
  const int t = threadIdx.x;
  const int64_t ncols = c.P * c.Q * c.J;
  const int64_t ntile = (ncols + kKgNT - 1) / kKgNT;
  const int nbg = op.BG > 0 ? op.BG : 1;
  const int64_t tile = blk % ntile, rest = blk / ntile;
  const int b0 = (int)(rest % nbg) * kKgMB;
  const int64_t split = rest / nbg;
  const int64_t i0 = split * op.chunk;
  const int64_t i1 = min(c.NI, i0 + op.chunk);
  const int NB = (int)c.NB;
  const int NBg = min(kKgMB, NB - b0);
  const bool rows = op.CG == 1;
  // load role, column-wise: column t of the tile, all kKgKT rows of a step;
  // row-wise: row t % 16 of columns t / 16 + 16 u
  const int lc = rows ? t / kKgKT : t, lr = rows ? t % kKgKT : 0;
  const float* in = (const float*)c.in;
  int64_t lbase = 0;
  bool lval = false;
  if (rows) {
    lbase = (tile * kKgNT + lc) * c.isP;
  } else {
    const I ln = (I)(tile * kKgNT + lc);
    lval = (int64_t)ln < ncols;
    if (lval) {
      const I j = ln % (I)c.J, pq = ln / (I)c.J;
      const I q = pq % (I)c.Q, p = pq / (I)c.Q;
      lbase = (int64_t)p * c.isP + (int64_t)q * c.isQ + (int64_t)j * c.isJ;
    }
  }
  const int64_t rstep = (int64_t)(kKgNT / kKgKT) * c.isP;   // row-wise: 16 columns on
  const int64_t rcols = ncols - tile * kKgNT;                // row-wise: valid columns
  // compute role: outputs b in [8 bg, 8 bg + 8), columns [4 cg, 4 cg + 4)
  const int cg = t % 64, bg = t / 64;
  float acc[8][4];
#pragma unroll
  for (int x = 0; x < 8; ++x)
#pragma unroll
    for (int y = 0; y < 4; ++y) acc[x][y] = 0.f;
  // the next step's rows are read into registers while this step computes
  constexpr int kRows = kKgKT * kKgNT / 256;      // tile entries each thread loads per step
  float ri[kRows], rw[kKgWPT];
#define KG_FETCH(k0_)                                                              \
  {                                                                                \
    const int nk_ = (int)min((int64_t)kKgKT, i1 - (k0_));                          \
    if (rows) {                                                                    \
      _Pragma("unroll") for (int u = 0; u < kRows; ++u)                            \
        ri[u] = (lr < nk_ && lc + u * (kKgNT / kKgKT) < rcols)                     \
                    ? in[lbase + u * rstep + (k0_) + lr] : 0.f;                    \
    } else {                                                                       \
      _Pragma("unroll") for (int u = 0; u < kRows; ++u)                            \
        ri[u] = (lval && u < nk_) ? in[lbase + ((k0_) + u) * c.isI] : 0.f;         \
    }                                                                              \
    _Pragma("unroll") for (int h = 0; h < kKgWPT; ++h) {                          \
      const int e_ = t + h * 256, kk_ = e_ / kKgMB, b_ = e_ % kKgMB;               \
      rw[h] = (b_ < NBg && kk_ < nk_) ? kg_weight(c, (k0_) + kk_, b0 + b_) : 0.f;  \
    }                                                                              \
  }
  if (i0 < i1) KG_FETCH(i0);
  for (int64_t k0 = i0; k0 < i1; k0 += kKgKT) {
    if (rows) {
#pragma unroll
      for (int u = 0; u < kRows; ++u) Is[lr * kKgLd + lc + u * (kKgNT / kKgKT)] = ri[u];
    } else {
#pragma unroll
      for (int u = 0; u < kRows; ++u) Is[u * kKgLd + lc] = ri[u];
    }
#pragma unroll
    for (int h = 0; h < kKgWPT; ++h) Ws[t + h * 256] = rw[h];
    __syncthreads();
    if (k0 + kKgKT < i1) KG_FETCH(k0 + kKgKT);
#pragma unroll
    for (int kk = 0; kk < kKgKT; ++kk) {
      const float4 w0 = *reinterpret_cast<const float4*>(&Ws[kk * kKgMB + 8 * bg]);
      const float4 w1 = *reinterpret_cast<const float4*>(&Ws[kk * kKgMB + 8 * bg + 4]);
      const float4 xv = *reinterpret_cast<const float4*>(&Is[kk * kKgLd + 4 * cg]);
#define KG_ROW(row_, w_)          \
  acc[row_][0] += (w_) * xv.x;    \
  acc[row_][1] += (w_) * xv.y;    \
  acc[row_][2] += (w_) * xv.z;    \
  acc[row_][3] += (w_) * xv.w;
      KG_ROW(0, w0.x) KG_ROW(1, w0.y) KG_ROW(2, w0.z) KG_ROW(3, w0.w)
      KG_ROW(4, w1.x) KG_ROW(5, w1.y) KG_ROW(6, w1.z) KG_ROW(7, w1.w)
#undef KG_ROW
    }
    __syncthreads();
  }
#undef KG_FETCH
#pragma unroll
  for (int y = 0; y < 4; ++y) {
    const I n = (I)(tile * kKgNT) + (I)(4 * cg + y);
    if ((int64_t)n >= ncols) continue;
    const I j = n % (I)c.J, pq = n / (I)c.J;
    const I q = pq % (I)c.Q, p = pq / (I)c.Q;
    // partial [split][p][b][q][j] or the output, at b = b0 + 8 bg
    const int64_t pbase = ((int64_t)split * c.P + p) * c.NB * c.Q * c.J + (int64_t)q * c.J + j;
    const int64_t pstep = c.Q * c.J;
    float* o = (float*)c.out + (int64_t)p * c.osP + (int64_t)q * c.osQ + (int64_t)j * c.osJ;
#pragma unroll
    for (int x = 0; x < 8; ++x) {
      const int b = b0 + 8 * bg + x;
      if (8 * bg + x >= NBg) continue;
      if (op.nsplit > 1) {
        ((float*)op.partial)[pbase + (int64_t)b * pstep] = acc[x][y];
      } else {
        float* ob = o + (int64_t)b * c.osB;
        const float v = (float)c.alpha * acc[x][y];
        *ob = c.accumulate ? *ob + v : v;
      }
    }
  }
}

template <typename I>
__device__ __forceinline__ I scatter_div(const Scatter& s, int a, I n) {
  if (sizeof(I) == 4) {
    const uint32_t r = (uint32_t)n;
    return (I)(uint32_t)(((uint64_t)__umulhi(r, s.mag[a]) + r) >> s.shf[a]);
  }
  return n / (I)s.size[a];
}

// Element e's offsets in `in` and `out` and its index on every scaled axis.
template <typename I>
__device__ __forceinline__ void scatter_decode(const Scatter& s, I e, int64_t* io, int64_t* oo,
                                               I* si) {
  int64_t ii = 0, o = 0;
  I rem = e;
  for (int a = s.nd - 1; a >= 0; --a) {
    const I q = scatter_div(s, a, rem);
    const I i = rem - q * (I)s.size[a];
    rem = q;
    ii += i * s.is[a];
    o += i * s.os[a];
#pragma unroll
    for (int k = 0; k < kMaxScales; ++k)
      if (k < s.nsc && s.scax[k] == a) si[k] = i;
  }
  *io = ii;
  *oo = o;
}

template <typename T, typename I>
__device__ void dev_scatter(const WalkOp& op, int64_t blk) {
  const Scatter& s = op.s;
  I total = 1;
  for (int a = 0; a < s.nd; ++a) total *= (I)s.size[a];
  // op.chunk elements per thread, kExecThreads apart: after the first, a
  // step stays on the last axis' row while it can (no full decode)
  const int L = s.nd - 1;
  const I nl = (I)s.size[L];
  const int64_t isl = s.is[L], osl = s.os[L];
  int lk = -1;   // the scale on the last axis, if any
  for (int k = 0; k < s.nsc; ++k)
    if (s.scax[k] == L) lk = k;
  I e = (I)(blk * op.chunk * kExecThreads) + (I)threadIdx.x;
  if (e >= total) return;
  int64_t io, oo;
  I si[kMaxScales];
#pragma unroll
  for (int k = 0; k < kMaxScales; ++k) si[k] = 0;
  scatter_decode(s, e, &io, &oo, si);
  I il = e - scatter_div(s, L, e) * nl;
  const T* in = (const T*)s.in;
  T* out = (T*)s.out;
  for (int it = 0;;) {
    T v = in[io];
#pragma unroll
    for (int k = 0; k < kMaxScales; ++k)
      if (k < s.nsc) v *= ((const T*)s.sc[k])[si[k]];
    if (s.assign) out[oo] = (T)s.alpha * v;
    else out[oo] = out[oo] + (T)s.alpha * v;
    if (++it == op.chunk) return;
    e += (I)kExecThreads;
    if (e >= total) return;
    il += (I)kExecThreads;
    if (il < nl) {
      io += (int64_t)kExecThreads * isl;
      oo += (int64_t)kExecThreads * osl;
      if (lk >= 0) {
#pragma unroll
        for (int k = 0; k < kMaxScales; ++k)
          if (k == lk) si[k] = il;
      }
    } else {
      scatter_decode(s, e, &io, &oo, si);
      il = e - scatter_div(s, L, e) * nl;
    }
  }
}

__device__ void dev_proj(const Proj& m, int64_t blk) {
  const int64_t e = blk * kExecThreads + threadIdx.x;
  if (e >= (int64_t)m.nq * m.ncols) return;
  const int q = (int)(e / m.ncols), j = (int)(e % m.ncols);
  const double* a = m.a + (int64_t)(m.q0 + q) * m.saq;
  double acc = 0.0;
  if (!m.F) {
    acc = a[(int64_t)j * m.sak];
  } else {
    const double* F = m.F + j;
    for (int64_t k = 0; k < m.n; ++k) acc += F[k * m.ldF] * a[k * m.sak];
  }
  if (m.has_w) acc *= m.w[q];
  m.out[(int64_t)q * m.ldo + j] = acc;
}

__device__ void dev_outer(const Outer& m, int64_t blk) {
  int64_t total = 1;
  for (int a = 0; a < m.A; ++a) total *= m.n[a];
  const int64_t e = blk * kExecThreads + threadIdx.x;
  if (e >= total) return;
  int64_t idx[kOuterAxes];
  int64_t rem = e, oo = 0;
  for (int a = m.A - 1; a >= 0; --a) {
    idx[a] = rem % m.n[a];
    rem /= m.n[a];
    oo += idx[a] * m.os[a];
  }
  int64_t xo[kOuterVecs];
  for (int k = 0; k < m.K; ++k) xo[k] = ((idx[m.ax[k]] / m.dv[k]) % m.md[k]) * m.si[k];
  double acc = 0.0;
  for (int q = 0; q < m.Q; ++q) {
    double t = 1.0;
    for (int k = 0; k < m.K; ++k) t *= m.v[k][(int64_t)q * m.sq[k] + xo[k]];
    acc += t;
  }
  if (m.out_f64) ((double*)m.out)[oo] += m.alpha * acc;
  else ((float*)m.out)[oo] += (float)(m.alpha * acc);
}

__device__ void dev_eye(const WalkOp& op, int64_t blk) {
  const int64_t n = op.eye_n;
  const int64_t e = blk * kExecThreads + threadIdx.x;
  if (e < n * n) ((double*)op.c.out)[e] = (e / n == e % n) ? 1.0 : 0.0;
}

// The op kinds of one accumulator type and index width.  Each (type, width)
// pair has a kernel of its own: a small level's time is mostly instruction
// fetch (16 to 20 stalled warps per issue before, with every kind, both types
// and both widths in one kernel), so a launch carries only the code its ops
// can reach.
template <bool F64, typename I>
__device__ __forceinline__ void dispatch(const WalkOp& op, int64_t blk, unsigned char* dsm) {
  typedef typename std::conditional<F64, double, float>::type T;
  switch (op.kind) {
    case OP_CONTRACT:
      if (!F64) dev_contract<T, T, T, T, I>(op, blk);
      else if (op.tin == ET_F64) dev_contract<double, double, double, double, I>(op, blk);
      else dev_contract<float, double, double, double, I>(op, blk);
      break;
    case OP_LANE:
      if (!F64) dev_lane<T, T, T, I>(op, blk, dsm);
      else if (op.tin == ET_F64) dev_lane<double, double, double, I>(op, blk, dsm);
      else dev_lane<float, double, double, I>(op, blk, dsm);
      break;
    case OP_SCATTER: dev_scatter<T, I>(op, blk); break;
    case OP_REDUCE: dev_reduce<T, I>(op, blk); break;
    case OP_EYE:
      if (F64) dev_eye(op, blk);
      break;
    case OP_MP:
      if (F64) break;   // binary64 products stay in the lane-group form
      if (op.CG == 0) {   // weight-stationary variant, NBT = op.BG
        switch (op.BG) {
          case 8: dev_mpw<8, I>(op, blk, dsm); break;
          case 16: dev_mpw<16, I>(op, blk, dsm); break;
          default: dev_mpw<32, I>(op, blk, dsm); break;
        }
      } else {
        dev_mp<float, I>(op, blk, dsm);
      }
      break;
    case OP_KRED:
      if (!F64) dev_kred(op, blk, dsm);
      break;
    default: break;
  }
}

// The op that holds block b, and b's place among its blocks.
template <typename Batch>
__device__ __forceinline__ int op_of_block(const Batch& lb, int b, int64_t* blk) {
  int lo = 0, hi = lb.nops - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) / 2;
    if (lb.start[mid] <= b) lo = mid;
    else hi = mid - 1;
  }
  *blk = b - lb.start[lo];
  return lo;
}

template <bool F64, typename I, int CAP>
__global__ void __launch_bounds__(kExecThreads, 3)
    level_kernel(const __grid_constant__ LevelBatch<WalkOp, CAP> lb) {
  extern __shared__ __align__(16) unsigned char dsm[];
  pdl_begin();
  int64_t blk;
  const int k = op_of_block(lb, (int)blockIdx.x, &blk);
  dispatch<F64, I>(lb.ops[k], blk, dsm);
}

// CP updates: projections and outer-product sums.
template <int CAP>
__global__ void __launch_bounds__(kExecThreads)
    cp_level_kernel(const __grid_constant__ LevelBatch<CpOp, CAP> lb) {
  pdl_begin();
  int64_t blk;
  const CpOp& op = lb.ops[op_of_block(lb, (int)blockIdx.x, &blk)];
  if (op.kind == OP_PROJ) dev_proj(op.pj, blk);
  else dev_outer(op.ou, blk);
}

// The split-K GEMM ops of a level in a kernel of their own (apart from the
// code of the other kinds).
// MINB resident blocks per SM: 2 (128 registers) for levels of a few waves,
// 3 (80 registers) for levels of many waves, where the extra warps hide more
// shared-memory latency and the coarser last wave costs little.
template <int MINB, int CAP>
__global__ void __launch_bounds__(kExecThreads, MINB)
    kgemm_level_kernel(const __grid_constant__ LevelBatch<WalkOp, CAP> lb) {
  extern __shared__ __align__(16) unsigned char dsm[];
  pdl_begin();
  int64_t blk;
  const int k = op_of_block(lb, (int)blockIdx.x, &blk);
  // one instantiation (64-bit column decoding: a few divisions per thread)
  dev_kgemm<int64_t>(lb.ops[k], blk, dsm);
}

// ---------------------------------------------------------------------------
// host parts
// ---------------------------------------------------------------------------
static bool mp_tiling(Op& op) {
  const Contract& c = op.c;
  if (!c.w || c.wsQ != 0 || c.wsJ != 0 || c.wsP != 0 || c.NI < 8 || c.NB > 64) return false;
  if (!(op.tin == op.tw && op.tw == op.tout)) return false;
  if (op.tout == ET_F64) return false;    // few FP64 units per SM: spread FP64 work thin instead
  if (c.P * c.Q * c.NB * c.J < 8192) return false;
  if (c.NI <= kWsMaxNI && c.NB <= 32) {
    // at most 32 outputs per thread (3 resident blocks per SM; wider weights
    // take the tiled form below)
    const int nbt = c.NB <= 8 ? 8 : c.NB <= 16 ? 16 : 32;
    op.kind = OP_MP;
    op.BG = nbt;
    op.CG = 0;
    op.CH = 0;
    op.blocks = ceil_div(c.P * c.Q * c.J, kExecThreads);
    return true;
  }
  int bg = (int)((c.NB + 3) / 4), p2 = 1;
  while (p2 < bg) p2 <<= 1;
  const int cg = std::min(kExecThreads / p2, 64);   // smem kMpKC2*4*(BG+CG)*4 <= 48 KB
  if (c.J > 4 * cg) return false;
  op.BG = p2;
  op.CG = cg;
  op.CH = (int)(4 * cg / c.J);
  const int64_t items = c.P * c.Q;
  op.blocks = ceil_div(items, op.CH);
  op.kind = OP_MP;
  return true;
}

int64_t plan_contract(Op& op) {
  op.kind = OP_CONTRACT;
  const Contract& c = op.c;
  const int64_t total = c.P * c.NB * c.Q * c.J;
  if (total == 0) {
    op.blocks = 0;
    return 0;
  }
  // split-K tiled form: b groups of kKgMB, long reductions split until the
  // blocks fill the GPU twice over (at least 64 reduction rows each)
  auto kgemm = [&]() -> int64_t {
    const int64_t ntile = ceil_div(c.P * c.Q * c.J, (int64_t)kKgNT);
    const int64_t nbg = ceil_div(c.NB, (int64_t)kKgMB);
    const int64_t want = (int64_t)exec_sms() * 2;
    // short reductions stay whole (the partial sums and their reduction
    // would cost more than the extra blocks gain)
    int64_t ns = c.NI < 1024 ? 1
                 : std::max<int64_t>(1, std::min<int64_t>(ceil_div(want, ntile * nbg), c.NI / 64));
    op.chunk = round_up(ceil_div(c.NI, ns), (int64_t)kKgKT);
    op.nsplit = (int)ceil_div(c.NI, op.chunk);
    op.kind = OP_KGEMM;
    op.BG = (int)nbg;
    // row-wise tile loads: one column per (p), contiguous reduction index
    op.CG = (c.J == 1 && c.Q == 1 && c.isI == 1 && c.P > 1) ? 1 : 0;
    op.blocks = ntile * nbg * op.nsplit;
    return op.nsplit > 1 ? total * op.nsplit : 0;
  };
  if (c.nkr > 0) {
    // Khatri-Rao weights exist only in the split-K tiled form (binary32,
    // NB <= kKgMB, weights independent of p, q, j: the recorder checks)
    return kgemm();
  }
  // long reductions with few outputs: split-K through shared-memory tiles
  if (c.w && c.wsQ == 0 && c.wsJ == 0 && c.wsP == 0 && op.tin == ET_F32 && op.tw == ET_F32 &&
      op.tout == ET_F32 && c.NI >= 2048 && c.NB <= 64 && c.J <= 64 &&
      c.NB * c.J <= 16 * kExecThreads && c.P * c.Q <= 64) {
    const int64_t items = c.P * c.Q;
    const int64_t want = (int64_t)exec_sms() * 4;
    int64_t ns = std::max<int64_t>(1, std::min<int64_t>(ceil_div(want, items), c.NI / kKredTile));
    op.chunk = round_up(ceil_div(c.NI, ns), kKredTile);
    op.nsplit = (int)ceil_div(c.NI, op.chunk);
    op.kind = OP_KRED;
    op.blocks = items * op.nsplit;
    return total * op.nsplit;
  }
  // the tiled and weight-stationary mode products give each thread many
  // outputs: for small ops that leaves most SMs idle while a few blocks run
  // long; there one lane group per output spreads the work instead
  const int64_t want = (int64_t)exec_sms() * 1024;   // threads that keep the GPU busy
  // binary32 mode products with reductions longer than the weight-stationary
  // form holds (e.g. a rank-200 TTN core against a sketch block) take the
  // split-K tiled form
  // (a product of few tiles would leave most SMs idle behind the latency of
  // its K steps: 24 tiles of 200 rows took 31 us; the lane form below spreads it)
  const bool few = ceil_div(c.P * c.Q * c.J, (int64_t)kKgNT) * ceil_div(c.NB, (int64_t)kKgMB) * 2 < exec_sms() &&
                   c.J >= 16 && c.isJ == 1;
  if (total >= want / 4 && c.w && c.wsQ == 0 && c.wsJ == 0 && c.wsP == 0 && c.NI > kWsMaxNI && !few &&
      c.NI < (int64_t(1) << 31) && op.tin == ET_F32 && op.tw == ET_F32 && op.tout == ET_F32)
    return kgemm();
  if (total >= want / 4 && mp_tiling(op)) return 0;
  // a contiguous output axis across the lanes, where a lane group per output
  // would cut the reduction index over the lanes of a warp
  const bool jl = c.J >= 4 && c.isJ == 1 && (!c.w || c.wsJ <= 1);
  const bool bl = c.J == 1 && c.NB >= 8 && c.w && c.wsB == 1;
  if ((jl || bl) && (total * 2 <= want || few) && c.NI >= 16) {
    const int64_t ln = jl ? c.J : c.NB;
    const int lw = ln <= 8 ? 8 : ln <= 16 ? 16 : 32;
    const int64_t units = (jl ? c.P * c.NB * c.Q : c.P * c.Q) * ceil_div(ln, (int64_t)lw);
    const int64_t warps = (int64_t)exec_sms() * 24;
    op.kind = OP_LANE;
    op.CH = jl ? 0 : 1;
    op.BG = lw;
    int ws = 1;
    while (ws < 8 && ceil_div(units, 32 / lw) * ws < warps && c.NI >= 16 * ws) ws <<= 1;
    op.CG = ws;
    int64_t ns = 1;
    if (c.NI >= 2048)
      ns = std::max<int64_t>(1, std::min<int64_t>(warps / (ceil_div(units, 32 / lw) * ws), c.NI / 512));
    op.chunk = ceil_div(c.NI, std::min<int64_t>(ns, 256));
    op.nsplit = (int)ceil_div(c.NI, op.chunk);
    op.blocks = ceil_div(ceil_div(units * op.nsplit, 32 / lw), 8 / ws);
    return op.nsplit > 1 ? total * op.nsplit : 0;
  }
  int g = 1;
  while (g < 32 && total * g < want && c.NI >= 8 * g) g <<= 1;
  op.g = g;
  op.nsplit = 1;
  op.chunk = c.NI;
  if (c.NI >= 2048 && total * g < want) {
    int64_t ns = std::min<int64_t>(ceil_div(want, total * g), c.NI / 512);
    ns = std::max<int64_t>(1, std::min<int64_t>(ns, 256));
    op.chunk = ceil_div(c.NI, ns);
    op.nsplit = (int)ceil_div(c.NI, op.chunk);
  }
  op.blocks = ceil_div(total * op.nsplit, kExecThreads / g);
  return op.nsplit > 1 ? total * op.nsplit : 0;
}

void plan_simple(Op& op) {
  int64_t total = 0;
  if (op.kind == OP_SCATTER) {
    total = 1;
    for (int a = 0; a < op.s.nd; ++a) total *= op.s.size[a];
    // large scatters: several elements per thread (fewer, fuller blocks)
    op.chunk = total >= (int64_t)exec_sms() * kExecThreads * 32 ? 8 : 1;
    op.blocks = ceil_div(total, (int64_t)kExecThreads * op.chunk);
    return;
  } else if (op.kind == OP_EYE) {
    total = op.eye_n * op.eye_n;
  } else if (op.kind == OP_REDUCE) {
    total = op.c.P * op.c.NB * op.c.Q * op.c.J;
  } else if (op.kind == OP_PROJ) {
    total = (int64_t)op.pj.nq * op.pj.ncols;
  } else if (op.kind == OP_OUTER) {
    total = 1;
    for (int a = 0; a < op.ou.A; ++a) total *= op.ou.n[a];
  }
  op.blocks = ceil_div(total, kExecThreads);
}

void Program::buffer(const void* p, int64_t bytes, int level) {
  if (!p || bytes <= 0) return;
  bufs_.push_back(Buf{(const char*)p, (const char*)p + bytes, level});
}

int Program::level_of(const void* p) const {
  if (!p) return 0;
  const char* c = (const char*)p;
  int lvl = 0;
  for (const Buf& b : bufs_)
    if (c >= b.lo && c < b.hi) lvl = std::max(lvl, b.level);
  return lvl;
}

void Program::add(Op op, const void* in1, const void* in2) {
  const int lvl = 1 + std::max(level_of(in1), level_of(in2));
  const void* out = op.kind == OP_SCATTER ? op.s.out
                    : op.kind == OP_PROJ  ? (const void*)op.pj.out
                    : op.kind == OP_OUTER ? op.ou.out
                                          : op.c.out;
  if (((op.kind == OP_CONTRACT || op.kind == OP_LANE || op.kind == OP_KGEMM) && op.nsplit > 1) ||
      op.kind == OP_KRED) {
    Op part = op;
    part.level = lvl;
    ops_.push_back(part);
    Op red = op;
    red.kind = OP_REDUCE;
    red.level = lvl + 1;
    plan_simple(red);
    ops_.push_back(red);
    for (Buf& b : bufs_)
      if ((const char*)out >= b.lo && (const char*)out < b.hi) b.level = std::max(b.level, lvl + 1);
    return;
  }
  op.level = lvl;
  ops_.push_back(op);
  for (Buf& b : bufs_)
    if ((const char*)out >= b.lo && (const char*)out < b.hi) b.level = std::max(b.level, lvl);
}

void Program::add(const TcOp& op, std::initializer_list<const void*> in) {
  int lvl = 0;
  for (const void* p : in) lvl = std::max(lvl, level_of(p));
  tcs_.push_back(op);
  tcs_.back().level = ++lvl;
  const char* out = (const char*)op.g.C;
  for (Buf& b : bufs_)
    if (out >= b.lo && out < b.hi) b.level = std::max(b.level, lvl);
}

// Debugging: runs what `launch` issues on `st` alone, synchronised, and prints
// its time.
template <typename Launch>
static ttnn_status timed_alone(cudaStream_t st, const Launch& launch) {
  cudaEvent_t a = nullptr, e = nullptr;
  TTNN_TRY_CUDA(cudaEventCreate(&a));
  TTNN_TRY_CUDA(cudaEventCreate(&e));
  TTNN_TRY_CUDA(cudaEventRecord(a, st));
  TTNN_TRY(launch());
  TTNN_TRY_CUDA(cudaEventRecord(e, st));
  TTNN_TRY_CUDA(cudaEventSynchronize(e));
  float ms = 0.f;
  cudaEventElapsedTime(&ms, a, e);
  cudaEventDestroy(a);
  cudaEventDestroy(e);
  fprintf(stderr, "[ttnn] %8.1f us  ", ms * 1e3f);
  return TTNN_OK;
}

static ttnn_status dump_tc(const TcOp& o, cudaStream_t st) {
  TcGemm g = o.g;
  g.prep = o.prep;
  TTNN_TRY(timed_alone(st, [&]() -> ttnn_status {
    void* const prep = o.prep;
    TTNN_TRY(tcg_prepare(&o.g, 1, &prep, st));
    return tcg_run(&g, 1, o.pieces, o.sms, o.err, o.wait_ns, st);
  }));
  fprintf(stderr, "[ttnn] L%d tensor-core gemm I %lld K %lld J %d type %d mn %d trans %d SMs %d\n", o.level,
          (long long)g.I, (long long)g.K, g.Jn, g.type, g.mn, g.trans, o.sms);
  return TTNN_OK;
}

// The tensor-core GEMMs of a level: their operands in one launch, then the
// products (those of several plans, with error words of their own, apart).
ttnn_status Program::run_tc(int lvl, cudaStream_t st, bool dump) const {
  for (const TcOp& o : tcs_)
    if (dump && o.level == lvl) TTNN_TRY(dump_tc(o, st));
  if (dump) return TTNN_OK;
  std::vector<TcGemm> g;
  std::vector<void*> prep;
  for (const TcOp& o : tcs_) {
    if (o.level != lvl) continue;
    g.push_back(o.g);
    prep.push_back(o.prep);
  }
  if (g.empty()) return TTNN_OK;
  TTNN_TRY(tcg_prepare(g.data(), (int)g.size(), prep.data(), st));
  const TcOp* first = nullptr;
  std::vector<TcGemm> run;
  auto flush = [&]() -> ttnn_status {
    if (run.empty()) return TTNN_OK;
    TTNN_TRY(tcg_run(run.data(), (int)run.size(), first->pieces, first->sms, first->err, first->wait_ns, st));
    run.clear();
    return TTNN_OK;
  };
  for (const TcOp& o : tcs_) {
    if (o.level != lvl) continue;
    if (run.empty()) first = &o;
    else if (o.pieces != first->pieces) {
      TTNN_TRY(flush());
      first = &o;
    }
    run.push_back(o.g);
    run.back().prep = o.prep;
  }
  return flush();
}

int Program::levels() const {
  int m = 0;
  for (const TcOp& o : tcs_) m = std::max(m, o.level);
  for (const Op& o : ops_) m = std::max(m, o.level);
  return m;
}

// Launch groups of a level: one kernel each.
enum LaunchGroup { LG_KGEMM = 0, LG_F32, LG_F32_WIDE, LG_F64, LG_F64_WIDE, LG_CP, LG_COUNT };

static LaunchGroup group_of(const Op& o) {
  if (o.kind == OP_KGEMM) return LG_KGEMM;
  if (o.kind == OP_PROJ || o.kind == OP_OUTER) return LG_CP;
  // 32-bit decoding when every extent and count stays below 2^31
  const int64_t lim = (int64_t(1) << 31) - 1;
  int64_t m = o.c.P * o.c.NB * o.c.Q * o.c.J * std::max(o.nsplit, 1);
  if (o.kind == OP_SCATTER) {
    int64_t st = 1;
    for (int a = 0; a < o.s.nd; ++a) st *= std::max<int64_t>(o.s.size[a], 1);
    m = std::max(m, st + (int64_t)kExecThreads * std::max<int64_t>(o.chunk, 1));
  }
  m = std::max(m, o.eye_n * o.eye_n);
  m = std::max(m, o.blocks * kExecThreads);
  if (o.tout == ET_F64) return m < lim ? LG_F64 : LG_F64_WIDE;
  return m < lim ? LG_F32 : LG_F32_WIDE;
}

static void to_dev(const Op& o, WalkOp* d) {
  d->kind = o.kind;
  d->tin = o.tin;
  if (o.kind == OP_SCATTER) d->s = o.s;
  else d->c = o.c;
  d->g = o.g;
  d->nsplit = o.nsplit;
  d->chunk = o.chunk;
  d->partial = o.partial;
  d->BG = o.BG;
  d->CG = o.CG;
  d->CH = o.CH;
  d->eye_n = o.eye_n;
}

static void to_dev(const Op& o, CpOp* d) {
  d->kind = o.kind;
  if (o.kind == OP_PROJ) d->pj = o.pj;
  else d->ou = o.ou;
}

template <typename OpT, int CAP>
static int64_t fill_batch(LevelBatch<OpT, CAP>& b, const Op* const* ops, int n) {
  b.nops = n;
  int64_t blocks = 0;
  for (int k = 0; k < n; ++k) {
    b.start[k] = (int)blocks;
    to_dev(*ops[k], &b.ops[k]);
    blocks += ops[k]->blocks;
    if (blocks >= (int64_t(1) << 31)) return -1;
  }
  b.start[n] = (int)blocks;
  return blocks;
}

template <int CAP>
static ttnn_status launch_group(LaunchGroup g, const Op* const* ops, int n, cudaStream_t st) {
  int64_t blocks;
  if (g == LG_CP) {
    LevelBatch<CpOp, CAP> b;
    if ((blocks = fill_batch(b, ops, n)) > 0)
      launch_pdl(cp_level_kernel<CAP>, (unsigned)blocks, kExecThreads, 0, st, b);
  } else {
    LevelBatch<WalkOp, CAP> b;
    blocks = fill_batch(b, ops, n);
    const unsigned gr = (unsigned)blocks;
    if (blocks <= 0) {
    } else if (g == LG_KGEMM) {
      // at least three full waves at three blocks per SM: the 80-register form
      if (blocks >= 9 * (int64_t)exec_sms())
        launch_pdl(kgemm_level_kernel<3, CAP>, gr, kExecThreads, kKgemmSmem, st, b);
      else
        launch_pdl(kgemm_level_kernel<2, CAP>, gr, kExecThreads, kKgemmSmem, st, b);
    } else if (g == LG_F32) {
      launch_pdl(level_kernel<false, uint32_t, CAP>, gr, kExecThreads, kExecSmem, st, b);
    } else if (g == LG_F32_WIDE) {
      launch_pdl(level_kernel<false, int64_t, CAP>, gr, kExecThreads, kExecSmem, st, b);
    } else if (g == LG_F64) {
      launch_pdl(level_kernel<true, uint32_t, CAP>, gr, kExecThreads, kLaneSmem, st, b);
    } else {
      launch_pdl(level_kernel<true, int64_t, CAP>, gr, kExecThreads, kLaneSmem, st, b);
    }
  }
  if (blocks < 0) {
    set_error("program level too large");
    return TTNN_EUNSUPPORTED;
  }
  if (blocks == 0) return TTNN_OK;
  return check_launch(g == LG_KGEMM ? "kgemm_level_kernel" : g == LG_CP ? "cp_level_kernel" : "level_kernel");
}

static ttnn_status launch_ops(LaunchGroup g, const std::vector<const Op*>& ops, cudaStream_t st) {
  for (size_t k = 0; k < ops.size(); k += kLargeOps) {
    const int n = (int)std::min<size_t>(ops.size() - k, kLargeOps);
    TTNN_TRY(n <= kSmallOps ? launch_group<kSmallOps>(g, ops.data() + k, n, st)
             : n <= kMidOps ? launch_group<kMidOps>(g, ops.data() + k, n, st)
                            : launch_group<kLargeOps>(g, ops.data() + k, n, st));
  }
  return TTNN_OK;
}

// A second stream per host thread and device for the split-K GEMM launches
// of a level, forked from and joined back into the caller's stream (so the
// two kernels of a level overlap; each thread keeps its own, so concurrent
// callers never wait on one another's work).
struct ForkStream {
  int device = -1;
  cudaStream_t st = nullptr;
  cudaEvent_t fork = nullptr, join = nullptr;
};

static ttnn_status fork_stream(ForkStream** out) {
  thread_local ForkStream fs[8];
  int dev = 0;
  TTNN_TRY_CUDA(cudaGetDevice(&dev));
  ForkStream* f = nullptr;
  for (auto& x : fs)
    if (x.device == dev) f = &x;
  if (!f) {
    for (auto& x : fs)
      if (x.device < 0) {
        f = &x;
        break;
      }
    if (!f) {
      *out = nullptr;   // more devices than slots: run the level's kernels in order
      return TTNN_OK;
    }
    TTNN_TRY_CUDA(cudaStreamCreateWithFlags(&f->st, cudaStreamNonBlocking));
    TTNN_TRY_CUDA(cudaEventCreateWithFlags(&f->fork, cudaEventDisableTiming));
    TTNN_TRY_CUDA(cudaEventCreateWithFlags(&f->join, cudaEventDisableTiming));
    f->device = dev;
  }
  *out = f;
  return TTNN_OK;
}

// Debugging: one op alone, timed (the stream is synchronised) and printed.
static ttnn_status dump_op(const Op& o, int lvl, cudaStream_t st) {
  TTNN_TRY(timed_alone(st, [&] { return launch_ops(group_of(o), {&o}, st); }));
  if (o.kind == OP_SCATTER)
    fprintf(stderr, "[ttnn] L%d scatter nd %d nsc %d blocks %lld\n", lvl, o.s.nd, o.s.nsc,
            (long long)o.blocks);
  else
    fprintf(stderr,
            "[ttnn] L%d kind %d P %lld NI %lld NB %lld Q %lld J %lld isJ %lld wsJ %lld "
            "wsQ %lld wsP %lld g %d nsplit %d blocks %lld\n",
            lvl, (int)o.kind, (long long)o.c.P, (long long)o.c.NI, (long long)o.c.NB,
            (long long)o.c.Q, (long long)o.c.J, (long long)o.c.isJ, (long long)o.c.wsJ,
            (long long)o.c.wsQ, (long long)o.c.wsP, o.g, o.nsplit, (long long)o.blocks);
  return TTNN_OK;
}

ttnn_status Program::run(cudaStream_t st, bool dump) {
  const int L = levels();
  // per level: the tensor-core GEMMs, the split-K GEMM ops in one launch of
  // their kernel, the other ops in one launch per type; when a level has
  // both, the GEMM launches go on the fork stream and run beside the others
  ForkStream* fs = nullptr;
  std::vector<const Op*> group[LG_COUNT];
  for (int lvl = 1; lvl <= L; ++lvl) {
    for (auto& g : group) g.clear();
    bool other = false;
    for (const Op& o : ops_) {
      if (o.level != lvl || o.blocks == 0) continue;
      if (dump) {
        TTNN_TRY(dump_op(o, lvl, st));
        continue;
      }
      const LaunchGroup g = group_of(o);
      group[g].push_back(&o);
      other = other || g != LG_KGEMM;
    }
    bool tc = false;
    for (const TcOp& o : tcs_) tc = tc || o.level == lvl;
    const bool fork = other && (tc || !group[LG_KGEMM].empty()) && !dump;
    cudaStream_t gst = st;   // stream of the GEMM launches
    if (fork) {
      if (!fs) TTNN_TRY(fork_stream(&fs));
      if (fs) {
        TTNN_TRY_CUDA(cudaEventRecord(fs->fork, st));
        TTNN_TRY_CUDA(cudaStreamWaitEvent(fs->st, fs->fork, 0));
        gst = fs->st;
      }
    }
    if (tc) TTNN_TRY(run_tc(lvl, gst, dump));
    for (int g = 0; g < LG_COUNT; ++g)
      if (!group[g].empty())
        TTNN_TRY(launch_ops((LaunchGroup)g, group[g], g == LG_KGEMM ? gst : st));
    if (gst != st) {
      TTNN_TRY_CUDA(cudaEventRecord(fs->join, gst));
      TTNN_TRY_CUDA(cudaStreamWaitEvent(st, fs->join, 0));
    }
  }
  return TTNN_OK;
}

}  // namespace ttnn
