// FP32 convolutions of the SIMT path (the plain FP32 form and the certifying pass) as implicit
// GEMMs: rows M = (subdomain row, output position), columns N = output channels, and K = (input
// channel, tap), the operand gathered from the channel-major FP32 activations while it is staged
// in shared memory.  The transposed convolution of the backward pass (Eq. definition_A) is split
// into its stride phases, as on the tensor-core path: input positions p = (a + s i, b + s j)
// receive only the taps ky = ky0(a) + s dy from source rows i + off(a) - dy, so no work is spent
// on the zeros of the stride and no thread diverges on a divisibility test.
//
// Each output is one sequential FMA chain over its K terms (K tile by K tile, in K order), at
// most the layer's terms_bwd / terms_fwd of them, so the certifying pass's a priori bound
// gamma_n sum |x_i y_i| (Higham, Accuracy and Stability of Numerical Algorithms, 3.1) holds.
#include <algorithm>
#include <atomic>
#include <mutex>
#include <vector>

#include "simt.cuh"

namespace bcrown {

extern std::atomic<long long> g_launches;

namespace {

struct SconvPass {
  uint32_t M;      // rows: R * Pm (below 2^31: a chunk's rows hold at least 12 Pm bytes each of 8 GB)
  int Pm, nJ;      // positions per row in this pass, and the pass grid's width
  FastDiv dPm, dnJ;
  int N, K;        // output channels; terms per output
  int Hs, Ws;      // source map (one channel)
  long long HWs;
  int ms, cy, cx;  // base source position of (i, j): (i ms + cy, j ms + cx)
  int oa, ob, os, Wo;
  long long HWo;   // output position (oa + os i) Wo + ob + os j, channel stride HWo
  const int4* tab; // [K]: {source offset c HWs + dy Ws + dx, dy, dx, tap = dy nkx + dx of the phase}
  const float* B;  // [K][N] weights
  int ky0, kx0;    // the phase's first tap (B depends on nothing else)
  int ntap;        // taps of the phase
  int nky, nkx;    // its rows and columns of taps, 0 in a forward pass
};
// A layer's stride phases, contracted by one launch.
constexpr int SC_PHASES = 4;
struct SconvPhases {
  SconvPass p[SC_PHASES];
};

// Rows of the output map that a row of the pass belongs to.
__device__ __forceinline__ long long sc_out(const SconvPass& q, uint32_t m, long long ostride, long long* pos) {
  const uint32_t rr = q.dPm(m);
  const int p2 = (int)(m - rr * (uint32_t)q.Pm);
  const int ii = (int)q.dnJ((uint32_t)p2), jj = p2 - ii * q.nJ;
  *pos = (long long)(q.oa + q.os * ii) * q.Wo + q.ob + q.os * jj;
  return (long long)rr * ostride + *pos;
}

// A 128 x BN tile, 8 x 8 outputs a thread (2 BN threads), FMAs on pairs of neighbouring channels
// (fma.rn.f32x2, as the GEMM), both operands by cp.async into two stages of 16 K terms: the
// gathered one in 4-byte pieces (a warp's are one run of positions), zero-filled where a tap falls
// outside the map, which is one bit per tap, worked out once a row.  Bound by the shared-memory pipe
// (48 % of its peak at 128 channels, 71 % at 32, where a gathered value feeds fewest FMAs) together
// with the FMA pipe; a third stage costs a resident block and is 3 % slower.  2,997 rows of the
// 32 -> 64 channel 4x4 stride-2 layer backward: 668 us in four launches with 8 x 2 outputs a thread
// and register staging, 420 with bounds tested per value and the lanes in row order, 335 now; 576
// rows of the 128 -> 128 channel 3x3 stride-2 layer 353 -> 271.
constexpr int SC_BM = 128, SC_BK = 16, SC_STAGES = 2;
constexpr int SC_AP = SC_BM + 4;

template <int BN>
__global__ void __launch_bounds__(2 * BN, BN == 32 ? 7 : 256 / BN)
    k_sconv(const SconvPhases ph, const float* __restrict__ src, long long sstride, float* __restrict__ out,
            long long ostride, const float* __restrict__ bias) {
  constexpr int NT = 2 * BN;
  constexpr int RPT = NT >= SC_BM ? 1 : SC_BM / NT;    // tile rows a thread gathers
  constexpr int KSTEP = NT >= SC_BM ? NT / SC_BM : 1;  // and the stride of its K terms
  const SconvPass& q = ph.p[blockIdx.z];
  const uint32_t m0 = blockIdx.x * (uint32_t)SC_BM;
  if (m0 >= q.M) return;
  extern __shared__ __align__(16) uint8_t sc_raw[];
  float* As = reinterpret_cast<float*>(sc_raw);                 // [stage][SC_BK][SC_AP]
  float* Bs = As + SC_STAGES * SC_BK * SC_AP;                   // [stage][SC_BK][BN]
  int2* stab = reinterpret_cast<int2*>(Bs + SC_STAGES * SC_BK * BN);   // [K, rounded up]: {offset, tap's bit}
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  // A warp's 32 threads are 8 row groups by 4 channel groups (16 by 2 where the block is one warp),
  // neighbouring lanes in the same row group: a 16-byte shared read then takes 2 wavefronts (4 with
  // the lanes in row order), and the shared pipe bounds the kernel beside the FMAs.
  const int ty = BN == 16 ? lane >> 1 : ((lane >> 1) & 7) + 8 * (w & 1);
  const int tx = BN == 16 ? lane & 1 : (lane & 1) + 2 * (lane >> 4) + 4 * (w >> 1);
  const int n0 = blockIdx.y * BN;
  const int nk = (q.K + SC_BK - 1) / SC_BK;
  const bool bits = q.ntap <= 32;
  for (int k = tid; k < nk * SC_BK; k += NT) {
    int2 e = make_int2(0, 0);
    if (k < q.K) {
      const int4 t = q.tab[k];
      e = make_int2(t.x, bits ? (int)(1u << t.w) : 0);
    }
    stab[k] = e;
  }
  // the rows this thread gathers (fixed across K), their base source positions and their taps in the map
  const float* srow[RPT];
  int pos[RPT], y0[RPT], x0[RPT];
  uint32_t inside[RPT];
#pragma unroll
  for (int u = 0; u < RPT; ++u) {
    const uint32_t m = m0 + (uint32_t)(tid % SC_BM) + (uint32_t)(u * NT);
    const bool mv = m < q.M;
    const uint32_t r = mv ? q.dPm(m) : 0u;
    const int pp = mv ? (int)(m - r * (uint32_t)q.Pm) : 0;
    const int pi = (int)q.dnJ((uint32_t)pp), pj = pp - pi * q.nJ;
    y0[u] = mv ? pi * q.ms + q.cy : -32768;
    x0[u] = pj * q.ms + q.cx;
    srow[u] = src + (long long)r * sstride;
    pos[u] = y0[u] * q.Ws + x0[u];
    inside[u] = 0u;
    for (int t = 0; bits && t < q.ntap; ++t) {
      const int4 e = q.tab[t];
      if ((unsigned)(y0[u] + e.y) < (unsigned)q.Hs && (unsigned)(x0[u] + e.z) < (unsigned)q.Ws) inside[u] |= 1u << t;
    }
  }
  const uint32_t sA = (uint32_t)__cvta_generic_to_shared(As), sB = (uint32_t)__cvta_generic_to_shared(Bs);
  const bool bvec = (q.N & 3) == 0;
  __syncthreads();
  auto load = [&](int stage, int k0) {
    const uint32_t as = sA + (uint32_t)(stage * SC_BK * SC_AP + tid % SC_BM) * 4;
    const uint32_t bs = sB + (uint32_t)(stage * SC_BK * BN) * 4;
    if (bits) {
#pragma unroll
      for (int k1 = 0; k1 < SC_BK; k1 += KSTEP) {
        const int kk = k1 + tid / SC_BM;
        const int2 t = stab[k0 + kk];
#pragma unroll
        for (int u = 0; u < RPT; ++u) {
          const bool in = (inside[u] & (uint32_t)t.y) != 0u;
          cp_async_fill<4>(as + (uint32_t)(kk * SC_AP + u * NT) * 4, srow[u] + (in ? pos[u] + t.x : 0), in ? 4 : 0);
        }
      }
    } else {
      for (int kk = tid / SC_BM; kk < SC_BK; kk += KSTEP) {
        const int k = k0 + kk;
        const int4 t = q.tab[min(k, q.K - 1)];
#pragma unroll
        for (int u = 0; u < RPT; ++u) {
          const bool in = k < q.K && (unsigned)(y0[u] + t.y) < (unsigned)q.Hs && (unsigned)(x0[u] + t.z) < (unsigned)q.Ws;
          cp_async_fill<4>(as + (uint32_t)(kk * SC_AP + u * NT) * 4, srow[u] + (in ? pos[u] + t.x : 0), in ? 4 : 0);
        }
      }
    }
    if (bvec) {
#pragma unroll
      for (int e0 = 0; e0 < SC_BK * (BN / 4); e0 += NT) {
        const int e = e0 + tid;   // (SC_BK BN / 4 = 2 NT)
        const int kk = e / (BN / 4), n = (e % (BN / 4)) * 4;
        const bool in = k0 + kk < q.K && n0 + n < q.N;
        cp_async_fill<16>(bs + (uint32_t)(kk * BN + n) * 4, in ? q.B + (size_t)(k0 + kk) * q.N + n0 + n : q.B,
                          in ? 16 : 0);
      }
    } else {
#pragma unroll
      for (int e0 = 0; e0 < SC_BK * BN; e0 += NT) {
        const int e = e0 + tid;
        const int kk = e / BN, n = e % BN;
        const bool in = k0 + kk < q.K && n0 + n < q.N;
        cp_async_fill<4>(bs + (uint32_t)(kk * BN + n) * 4, in ? q.B + (size_t)(k0 + kk) * q.N + n0 + n : q.B,
                         in ? 4 : 0);
      }
    }
  };
  // thread (ty, tx): rows 4 ty .. + 3 and 64 + 4 ty .. + 3, channels 4 tx .. + 3 of each half
  unsigned long long acc[8][4];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0ull;
#pragma unroll
  for (int t = 0; t < SC_STAGES - 1; ++t) {
    if (t < nk) load(t, t * SC_BK);
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  int st = 0, ld = SC_STAGES - 1;
  for (int t = 0; t < nk; ++t) {
    asm volatile("cp.async.wait_group %0;" ::"n"(SC_STAGES - 2) : "memory");
    __syncthreads();
    if (t + SC_STAGES - 1 < nk) load(ld, (t + SC_STAGES - 1) * SC_BK);
    asm volatile("cp.async.commit_group;" ::: "memory");
    const float* as = As + st * SC_BK * SC_AP + 4 * ty;
    const float* bs = Bs + st * SC_BK * BN + 4 * tx;
    if (++st == SC_STAGES) st = 0;
    if (++ld == SC_STAGES) ld = 0;
#pragma unroll
    for (int kk = 0; kk < SC_BK; ++kk) {
      const float4 a0 = *reinterpret_cast<const float4*>(as + kk * SC_AP);
      const float4 a1 = *reinterpret_cast<const float4*>(as + kk * SC_AP + 64);
      const ulonglong2 b0 = *reinterpret_cast<const ulonglong2*>(bs + kk * BN);
      const ulonglong2 b1 = *reinterpret_cast<const ulonglong2*>(bs + kk * BN + BN / 2);
      const float av[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const unsigned long long a = f32x2_dup(av[i]);
        f32x2_fma(acc[i][0], a, b0.x);
        f32x2_fma(acc[i][1], a, b0.y);
        f32x2_fma(acc[i][2], a, b1.x);
        f32x2_fma(acc[i][3], a, b1.y);
      }
    }
  }
  // four neighbouring rows are four neighbouring outputs where the pass covers whole map rows
  const bool v4 = q.os == 1 && ((q.nJ | q.Wo) & 3) == 0 && (q.ob & 3) == 0 && ((q.HWo | ostride) & 3) == 0 &&
                  ((reinterpret_cast<uintptr_t>(out) | reinterpret_cast<uintptr_t>(bias)) & 15) == 0;
#pragma unroll
  for (int hm = 0; hm < 2; ++hm) {
    const uint32_t mb = m0 + 64u * hm + 4u * ty;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int n = n0 + (j < 4 ? 4 * tx + j : BN / 2 + 4 * tx + j - 4);
      if (n >= q.N) continue;
      float o[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float2 x = f32x2_split(acc[4 * hm + i][j / 2]);
        o[i] = j & 1 ? x.y : x.x;
      }
      if (v4 && mb + 3 < q.M) {
        long long pos;
        float* op = out + sc_out(q, mb, ostride, &pos) + (size_t)n * q.HWo;
        float4 b = make_float4(0.f, 0.f, 0.f, 0.f);
        if (bias) b = *reinterpret_cast<const float4*>(bias + (size_t)n * q.HWo + pos);
        *reinterpret_cast<float4*>(op) = make_float4(o[0] + b.x, o[1] + b.y, o[2] + b.z, o[3] + b.w);
      } else {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          if (mb + i >= q.M) continue;
          long long pos;
          const long long at = sc_out(q, mb + i, ostride, &pos);
          out[at + n * q.HWo] = o[i] + (bias ? bias[(size_t)n * q.HWo + pos] : 0.f);
        }
      }
    }
  }
}

// Passes with at most 4 output channels (the backward pass of a first layer over 1-4 input
// channels): a 128 x 16 tile would spend most of its FMAs on padding and its shared-memory reads
// would outnumber them, and no operand value is reused across output channels anyway.  Each
// thread computes 4 rows (m, m + 256, m + 512, m + 768 of its block, so every load of a warp is
// one contiguous run of positions) times the N channels, loading its operand straight from
// global memory; the K loop reads the tap table and the N weights of each term from shared
// memory (one broadcast load each).  Each output is the same sequential FMA chain in K order as
// in k_sconv, so the result is the same bit for bit and the same a priori error bound holds.
//
// Which taps of a row lie inside the map is one bit each, worked out once, and 8 terms' loads (32 a
// thread) are in flight together: with the bounds tested per term and 2 terms at a time the kernel
// waited for its loads three quarters of the time.  All stride phases are one launch.  Layers whose taps
// share a window go to k_sconv_cells.
constexpr int SN_THREADS = 256, SN_TM = 4;

template <int N>
__global__ void __launch_bounds__(SN_THREADS) k_sconv_narrow(const SconvPhases ph, const float* __restrict__ src,
                                                            long long sstride, float* __restrict__ out,
                                                            long long ostride, const float* __restrict__ bias) {
  const SconvPass& q = ph.p[blockIdx.z];
  if (blockIdx.x * (uint32_t)(SN_THREADS * SN_TM) >= q.M) return;
  extern __shared__ __align__(16) uint8_t sn_raw[];
  int4* stab = reinterpret_cast<int4*>(sn_raw);
  float4* sB = reinterpret_cast<float4*>(sn_raw + (size_t)q.K * sizeof(int4));
  const int tid = threadIdx.x;
  for (int k = tid; k < q.K; k += SN_THREADS) {
    stab[k] = q.tab[k];
    const float* b = q.B + (size_t)k * N;
    sB[k] = make_float4(b[0], N > 1 ? b[1] : 0.f, N > 2 ? b[2] : 0.f, N > 3 ? b[3] : 0.f);
  }
  __syncthreads();
  const float* srow[SN_TM];
  uint32_t inside[SN_TM];   // taps inside the map (the first 32; the others are tested per term)
  int y0[SN_TM], x0[SN_TM];
#pragma unroll
  for (int i = 0; i < SN_TM; ++i) {
    const uint32_t m = blockIdx.x * (uint32_t)(SN_THREADS * SN_TM) + i * SN_THREADS + tid;
    const bool mv = m < q.M;
    const uint32_t r = mv ? q.dPm(m) : 0u;
    const int pp = mv ? (int)(m - r * (uint32_t)q.Pm) : 0;
    const int pi = (int)q.dnJ((uint32_t)pp), pj = pp - pi * q.nJ;
    y0[i] = mv ? pi * q.ms + q.cy : -32768;
    x0[i] = pj * q.ms + q.cx;
    srow[i] = src + (long long)r * sstride + (mv ? (long long)y0[i] * q.Ws + x0[i] : 0);
    inside[i] = 0u;
    for (int t = 0; t < min(q.ntap, 32); ++t)
      if ((unsigned)(y0[i] + stab[t].y) < (unsigned)q.Hs && (unsigned)(x0[i] + stab[t].z) < (unsigned)q.Ws)
        inside[i] |= 1u << t;
  }
  float acc[SN_TM][N];
#pragma unroll
  for (int i = 0; i < SN_TM; ++i)
#pragma unroll
    for (int j = 0; j < N; ++j) acc[i][j] = 0.f;
  if (q.ntap <= 32) {
    constexpr int KU = 8;
    for (int k0 = 0; k0 < q.K; k0 += KU) {
      float v[KU][SN_TM];
#pragma unroll
      for (int e = 0; e < KU; ++e) {
        const int k = min(k0 + e, q.K - 1);
        const int2 t = make_int2(stab[k].x, k0 + e < q.K ? stab[k].w : 32);
#pragma unroll
        for (int i = 0; i < SN_TM; ++i) {
          v[e][i] = 0.f;
          if (t.y < 32 && (inside[i] >> t.y) & 1u) v[e][i] = srow[i][t.x];
        }
      }
#pragma unroll
      for (int e = 0; e < KU; ++e) {
        if (k0 + e >= q.K) break;
        const float4 b4 = sB[k0 + e];
        const float bv[4] = {b4.x, b4.y, b4.z, b4.w};
#pragma unroll
        for (int i = 0; i < SN_TM; ++i)
#pragma unroll
          for (int j = 0; j < N; ++j) acc[i][j] = fmaf(v[e][i], bv[j], acc[i][j]);
      }
    }
  } else {
    for (int k = 0; k < q.K; ++k) {
      const int4 t = stab[k];
      const float4 b4 = sB[k];
      const float bv[4] = {b4.x, b4.y, b4.z, b4.w};
#pragma unroll
      for (int i = 0; i < SN_TM; ++i) {
        const bool in = (unsigned)(y0[i] + t.y) < (unsigned)q.Hs && (unsigned)(x0[i] + t.z) < (unsigned)q.Ws;
        const float v = in ? srow[i][t.x] : 0.f;
#pragma unroll
        for (int j = 0; j < N; ++j) acc[i][j] = fmaf(v, bv[j], acc[i][j]);
      }
    }
  }
#pragma unroll
  for (int i = 0; i < SN_TM; ++i) {
    const uint32_t m = blockIdx.x * (uint32_t)(SN_THREADS * SN_TM) + i * SN_THREADS + tid;
    if (m >= q.M) continue;
    long long p;
    float* orow = out + sc_out(q, m, ostride, &p);
#pragma unroll
    for (int j = 0; j < N; ++j) orow[(size_t)j * q.HWo] = acc[i][j] + (bias ? bias[(size_t)j * q.HWo + p] : 0.f);
  }
}

// The common first layers' backward pass (3x3 stride 1, 4x4 stride 2; at most 4 input channels): a
// thread takes cells of 2 x 2 outputs, whose taps lie in one (T + SH) x (T + SH) window of the source,
// so a value is loaded once for the outputs that share it (9 loads a channel instead of 16 with 4x4
// stride 2, 16 instead of 36 with 3x3): k_sconv_narrow is bound by its loads and what surrounds them.
// Output (2 i + a, 2 j + b), tap (dy, dx) reads window row SH a + T - 1 - dy and column SH b + T - 1 - dx:
// T = 3, SH = 1 for 3x3 stride 1, T = 2 for 4x4 stride 2 with SH the padding's parity.  Every output's
// sum has the order of the general pass.  2,997 rows of 3 x 32 x 32 from 32 channels (4x4 stride 2):
// k_sconv_narrow 183 us, here 109; 576 rows from 64 channels (3x3) 169 / 83; 1,024 rows of 18 x 18
// patches (padding 0) 57 / 28.
struct SconvCells {
  uint32_t M;        // cells of all rows
  int Pm, nJ;        // cells of a row, and of a row of cells
  FastDiv dPm, dnJ;
  int Hs, Ws, C;     // source map, its channels
  long long HWs;
  int ms, cy, cx;    // window origin of cell (i, j): (i ms + cy, j ms + cx)
  int Ho, Wo;
  long long HWo;
  const float* B[4]; // [C T T][N] weights of output (a, b) of a cell, at 2 a + b (stride 1: one for all)
};
constexpr int SL_THREADS = 128, SL_CELLS = 2;   // cells a thread

template <int N, int T, int SH>
__global__ void __launch_bounds__(SL_THREADS) k_sconv_cells(const SconvCells q, const float* __restrict__ src,
                                                           long long sstride, float* __restrict__ out,
                                                           long long ostride) {
  constexpr int W = T + SH, TT = T * T, NP = T == 3 ? 1 : 4;
  extern __shared__ __align__(16) uint8_t sl_raw[];
  float4* sB = reinterpret_cast<float4*>(sl_raw);   // [C][NP][T T]
  for (int e = threadIdx.x; e < q.C * NP * TT; e += SL_THREADS) {
    const int t = e % TT, ph = e / TT % NP, c = e / (TT * NP);
    const float* b = (ph == 0 ? q.B[0] : ph == 1 ? q.B[1] : ph == 2 ? q.B[2] : q.B[3]) + (size_t)(c * TT + t) * N;
    sB[e] = make_float4(b[0], N > 1 ? b[1] : 0.f, N > 2 ? b[2] : 0.f, N > 3 ? b[3] : 0.f);
  }
  __syncthreads();
  const float* win[SL_CELLS];
  uint32_t in[SL_CELLS];
  long long at[SL_CELLS];
  int edge[SL_CELLS];   // bit 0: a second row of outputs, bit 1: a second column, bit 2: any
#pragma unroll
  for (int u = 0; u < SL_CELLS; ++u) {
    const uint32_t m = blockIdx.x * (uint32_t)(SL_THREADS * SL_CELLS) + u * SL_THREADS + threadIdx.x;
    const bool mv = m < q.M;
    const uint32_t r = mv ? q.dPm(m) : 0u;
    const int pp = mv ? (int)(m - r * (uint32_t)q.Pm) : 0;
    const int ci = (int)q.dnJ((uint32_t)pp), cj = pp - ci * q.nJ;
    const int y0 = ci * q.ms + q.cy, x0 = cj * q.ms + q.cx;
    win[u] = src + (long long)r * sstride + ((long long)y0 * q.Ws + x0);
    in[u] = 0u;
#pragma unroll
    for (int y = 0; y < W; ++y)
#pragma unroll
      for (int x = 0; x < W; ++x)
        if (mv && (unsigned)(y0 + y) < (unsigned)q.Hs && (unsigned)(x0 + x) < (unsigned)q.Ws) in[u] |= 1u << (y * W + x);
    at[u] = (long long)r * ostride + (long long)(2 * ci) * q.Wo + 2 * cj;
    edge[u] = mv ? 4 | (2 * ci + 1 < q.Ho ? 1 : 0) | (2 * cj + 1 < q.Wo ? 2 : 0) : 0;
  }
  float acc[SL_CELLS][4][N];
#pragma unroll
  for (int u = 0; u < SL_CELLS; ++u)
#pragma unroll
    for (int o = 0; o < 4; ++o)
#pragma unroll
      for (int n = 0; n < N; ++n) acc[u][o][n] = 0.f;
  for (int c = 0; c < q.C; ++c) {
    float v[SL_CELLS][W * W];
#pragma unroll
    for (int u = 0; u < SL_CELLS; ++u) {
#pragma unroll
      for (int y = 0; y < W; ++y) {
        const float* row = win[u] + (long long)y * q.Ws;
#pragma unroll
        for (int x = 0; x < W; ++x) {
          v[u][y * W + x] = 0.f;
          if ((in[u] >> (y * W + x)) & 1u) v[u][y * W + x] = row[x];
        }
      }
      win[u] += q.HWs;
    }
    const float4* wc = sB + c * NP * TT;
#pragma unroll
    for (int ph = 0; ph < NP; ++ph)
#pragma unroll
      for (int dy = 0; dy < T; ++dy)
#pragma unroll
        for (int dx = 0; dx < T; ++dx) {
          const float4 b4 = wc[ph * TT + dy * T + dx];
          const float bv[4] = {b4.x, b4.y, b4.z, b4.w};
#pragma unroll
          for (int o = 0; o < 4; ++o) {
            if (NP == 4 && o != ph) continue;
            const int a = o >> 1, b = o & 1;
            const int e = (SH * a + T - 1 - dy) * W + SH * b + T - 1 - dx;
#pragma unroll
            for (int u = 0; u < SL_CELLS; ++u)
#pragma unroll
              for (int n = 0; n < N; ++n) acc[u][o][n] = fmaf(v[u][e], bv[n], acc[u][o][n]);
          }
        }
  }
  const bool pairs = ((q.Wo | (int)(q.HWo & 1) | (int)(ostride & 1)) & 1) == 0 &&
                     (reinterpret_cast<uintptr_t>(out) & 7) == 0;
#pragma unroll
  for (int u = 0; u < SL_CELLS; ++u) {
    if (!edge[u]) continue;
#pragma unroll
    for (int n = 0; n < N; ++n)
#pragma unroll
      for (int a = 0; a < 2; ++a) {
        if (a && !(edge[u] & 1)) continue;
        float* o = out + at[u] + n * q.HWo + (long long)a * q.Wo;
        if (pairs) {
          *reinterpret_cast<float2*>(o) = make_float2(acc[u][2 * a][n], acc[u][2 * a + 1][n]);
        } else {
          o[0] = acc[u][2 * a][n];
          if (edge[u] & 2) o[1] = acc[u][2 * a + 1][n];
        }
      }
  }
}

constexpr int SL_SMEM = 96 * 1024;
int sconv_cells_smem(int C, int T) { return C * (T == 3 ? 9 : 16) * (int)sizeof(float4); }

template <int T, int SH>
cudaError_t cells_attr() {
  cudaError_t e = cudaFuncSetAttribute(k_sconv_cells<1, T, SH>, cudaFuncAttributeMaxDynamicSharedMemorySize, SL_SMEM);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_sconv_cells<2, T, SH>, cudaFuncAttributeMaxDynamicSharedMemorySize, SL_SMEM);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_sconv_cells<3, T, SH>, cudaFuncAttributeMaxDynamicSharedMemorySize, SL_SMEM);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_sconv_cells<4, T, SH>, cudaFuncAttributeMaxDynamicSharedMemorySize, SL_SMEM);
  return e;
}

int sconv_narrow_smem(int K) { return K * (int)(sizeof(int4) + sizeof(float4)); }

int sconv_smem(int BN, int K) {
  return SC_STAGES * SC_BK * (SC_AP + BN) * 4 + (K + SC_BK - 1) / SC_BK * SC_BK * (int)sizeof(int2);
}

struct LayerF32 {
  std::vector<SconvPass> bwd;   // one per stride phase with positions
  SconvPass fwd;
  // [T]: the backward passes over the patches of layer T's root rows (root.cu)
  std::vector<std::vector<SconvPass>> patch;
};
struct SconvNet {
  bool ready = false;
  std::vector<LayerF32> ly;     // ly[i]: paper layer i (conv layers only)
  std::vector<void*> bufs;
};

std::mutex g_sc_mu;
std::vector<std::pair<const bcrown_net*, SconvNet*>> g_sc;

SconvNet* sc_of(const bcrown_net* net) {
  std::lock_guard<std::mutex> g(g_sc_mu);
  for (auto& e : g_sc)
    if (e.first == net) return e.second;
  SconvNet* t = new SconvNet();
  g_sc.push_back({net, t});
  return t;
}

int sc_upload(SconvNet* t, const void* host, size_t bytes, void** dev) {
  if (cudaMalloc(dev, bytes) != cudaSuccess) return fail(BCROWN_ERR_OOM, "FP32 conv: device tables");
  t->bufs.push_back(*dev);
  if (cudaMemcpy(*dev, host, bytes, cudaMemcpyHostToDevice) != cudaSuccess)
    return fail(BCROWN_ERR_CUDA, "FP32 conv: table upload");
  return BCROWN_OK;
}

// Phase a of one spatial axis of a stride-s transposed convolution: the taps k0 + s d (d < nk)
// reach input rows a + s i (i < n), whose source row is i + off - d.
void sc_phase(int a, int k, int s, int pad, int in, int* k0, int* nk, int* off, int* n) {
  *k0 = (a + pad) % s;
  *nk = *k0 < k ? (k - *k0 + s - 1) / s : 0;
  *off = (a + pad - *k0) / s;
  *n = a < in ? (in - a + s - 1) / s : 0;
}

int sc_prepare(bcrown_net* net, SconvNet* t) {
  if (t->ready) return BCROWN_OK;
  t->ly.assign(net->L, LayerF32());
  bool any = false;
  for (int i = 1; i <= net->L - 1; ++i) {
    const LayerDev& l = net->ly[i - 1];
    if (!sconv_supported(net, i)) continue;
    any = true;
    const int k = l.k, s = l.stride, kk = k * k;
    std::vector<float> w((size_t)l.out_c * l.in_c * kk);
    if (cudaMemcpy(w.data(), l.W, w.size() * 4, cudaMemcpyDeviceToHost) != cudaSuccess)
      return fail(BCROWN_ERR_CUDA, "FP32 conv: copy of weights");
    LayerF32& P = t->ly[i];
    // backward phases: source Lambda^(i) (out_c x out_h x out_w), output the input map
    auto backward = [&](int in_h, int in_w, int out_h, int out_w, int pad, std::vector<SconvPass>& made) -> int {
    for (int a = 0; a < s; ++a)
      for (int b = 0; b < s; ++b) {
        int ky0, nky, offy, ny, kx0, nkx, offx, nx;
        sc_phase(a, k, s, pad, in_h, &ky0, &nky, &offy, &ny);
        sc_phase(b, k, s, pad, in_w, &kx0, &nkx, &offx, &nx);
        if (ny * nx == 0) continue;
        SconvPass q{};
        q.Pm = ny * nx;
        q.nJ = nx;
        q.N = l.in_c;
        q.K = std::max(1, l.out_c * nky * nkx);
        q.Hs = out_h;
        q.Ws = out_w;
        q.HWs = (long long)out_h * out_w;
        q.ms = 1;
        q.cy = offy;
        q.cx = offx;
        q.oa = a;
        q.ob = b;
        q.os = s;
        q.Wo = in_w;
        q.HWo = (long long)in_h * in_w;
        q.ky0 = ky0;
        q.kx0 = kx0;
        q.ntap = std::max(1, nky * nkx);
        q.nky = nky;
        q.nkx = nkx;
        q.dPm.set(q.Pm);
        q.dnJ.set(q.nJ);
        std::vector<int4> tab((size_t)q.K, make_int4(0, -32768, 0, 0));
        for (int co = 0; co < l.out_c; ++co)
          for (int dy = 0; dy < nky; ++dy)
            for (int dx = 0; dx < nkx; ++dx)
              tab[(co * nky + dy) * nkx + dx] = make_int4((int)(co * q.HWs - dy * out_w - dx), -dy, -dx, dy * nkx + dx);
        void *dt = nullptr, *dB = nullptr;
        BC_CHECK(sc_upload(t, tab.data(), tab.size() * sizeof(int4), &dt));
        q.tab = reinterpret_cast<const int4*>(dt);
        for (const SconvPass& o : P.bwd)   // the phase's weights, if another pass of the layer has them
          if (o.ky0 == ky0 && o.kx0 == kx0) q.B = o.B;
        if (!q.B) {
          std::vector<float> B((size_t)q.K * q.N, 0.f);
          for (int co = 0; co < l.out_c; ++co)
            for (int dy = 0; dy < nky; ++dy)
              for (int dx = 0; dx < nkx; ++dx) {
                const int kq = (co * nky + dy) * nkx + dx, ky = ky0 + s * dy, kx = kx0 + s * dx;
                for (int ci = 0; ci < l.in_c; ++ci)
                  B[(size_t)kq * q.N + ci] = w[(((size_t)co * l.in_c + ci) * k + ky) * k + kx];
              }
          BC_CHECK(sc_upload(t, B.data(), B.size() * 4, &dB));
          q.B = reinterpret_cast<const float*>(dB);
        }
        made.push_back(q);
      }
      return BCROWN_OK;
    };
    BC_CHECK(backward(l.in_h, l.in_w, l.out_h, l.out_w, l.pad, P.bwd));
    P.patch.assign(net->L, std::vector<SconvPass>());
    for (int T = i + 1; T <= net->L - 1; ++T) {
      std::vector<int> n;
      if (root_patch(net, T, n)) BC_CHECK(backward(n[i - 1], n[i - 1], n[i], n[i], 0, P.patch[T]));
    }
    // forward: source h^(i-1) (in_c x in_h x in_w), output the layer's map
    SconvPass f{};
    f.Pm = l.out_h * l.out_w;
    f.nJ = l.out_w;
    f.N = l.out_c;
    f.K = l.in_c * kk;
    f.Hs = l.in_h;
    f.Ws = l.in_w;
    f.HWs = (long long)l.in_h * l.in_w;
    f.ms = s;
    f.cy = -l.pad;
    f.cx = -l.pad;
    f.oa = 0;
    f.ob = 0;
    f.os = 1;
    f.Wo = l.out_w;
    f.HWo = (long long)l.out_h * l.out_w;
    f.ntap = kk;
    f.dPm.set(f.Pm);
    f.dnJ.set(f.nJ);
    std::vector<int4> tab((size_t)f.K);
    std::vector<float> B((size_t)f.K * f.N);
    for (int ci = 0; ci < l.in_c; ++ci)
      for (int ky = 0; ky < k; ++ky)
        for (int kx = 0; kx < k; ++kx) {
          const int kq = (ci * k + ky) * k + kx;
          tab[kq] = make_int4((int)(ci * f.HWs + ky * l.in_w + kx), ky, kx, ky * k + kx);
          for (int co = 0; co < l.out_c; ++co) B[(size_t)kq * f.N + co] = w[(((size_t)co * l.in_c + ci) * k + ky) * k + kx];
        }
    void *dt = nullptr, *dB = nullptr;
    BC_CHECK(sc_upload(t, tab.data(), tab.size() * sizeof(int4), &dt));
    BC_CHECK(sc_upload(t, B.data(), B.size() * 4, &dB));
    f.tab = reinterpret_cast<const int4*>(dt);
    f.B = reinterpret_cast<const float*>(dB);
    P.fwd = f;
  }
  if (!any) {   // (the attributes below load every kernel, which a net without convolutions need not wait for)
    t->ready = true;
    return BCROWN_OK;
  }
  {
    const int smem = sconv_narrow_smem(SCONV_MAX_K);
    for (cudaError_t e : {cudaFuncSetAttribute(k_sconv_narrow<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem),
                          cudaFuncSetAttribute(k_sconv_narrow<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem),
                          cudaFuncSetAttribute(k_sconv_narrow<3>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem),
                          cudaFuncSetAttribute(k_sconv_narrow<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem)})
      if (e != cudaSuccess)
        return fail(BCROWN_ERR_CUDA, std::string("FP32 conv: smem attribute: ") + cudaGetErrorString(e));
  }
  for (cudaError_t e : {cells_attr<3, 1>(), cells_attr<2, 1>(), cells_attr<2, 0>()})
    if (e != cudaSuccess)
      return fail(BCROWN_ERR_CUDA, std::string("FP32 conv: smem attribute: ") + cudaGetErrorString(e));
  for (int BN : {16, 32, 64, 128}) {
    const int smem = sconv_smem(BN, SCONV_MAX_K);
    cudaError_t e = BN == 16    ? cudaFuncSetAttribute(k_sconv<16>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem)
                    : BN == 32  ? cudaFuncSetAttribute(k_sconv<32>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem)
                    : BN == 64  ? cudaFuncSetAttribute(k_sconv<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem)
                                : cudaFuncSetAttribute(k_sconv<128>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return fail(BCROWN_ERR_CUDA, std::string("FP32 conv: smem attribute: ") + cudaGetErrorString(e));
  }
  t->ready = true;
  return BCROWN_OK;
}

template <int T, int SH>
void cells_launch(int N, unsigned grid, int smem, const SconvCells& c, const float* src, long long sstride, float* out,
                  long long ostride, cudaStream_t s) {
  auto go = [&](auto* k) { k<<<grid, SL_THREADS, smem, s>>>(c, src, sstride, out, ostride); };
  if (N == 1) go(k_sconv_cells<1, T, SH>);
  else if (N == 2) go(k_sconv_cells<2, T, SH>);
  else if (N == 3) go(k_sconv_cells<3, T, SH>);
  else go(k_sconv_cells<4, T, SH>);
}

// A backward contraction that the cells' kernel takes (its geometry is in the passes); false: it does not.
bool cells_try(const SconvPass* q, int n, int R, const float* src, long long sstride, float* out, long long ostride,
               cudaStream_t s) {
  if (q[0].N > 4) return false;
  const bool s1 = n == 1 && q[0].os == 1 && q[0].nky == 3 && q[0].nkx == 3;
  bool s2 = n == 4 && q[0].os == 2;
  for (int z = 0; s2 && z < 4; ++z) s2 = q[z].nky == 2 && q[z].nkx == 2 && q[z].oa == z / 2 && q[z].ob == z % 2;
  if (!s1 && !s2) return false;
  const int T = s1 ? 3 : 2, SH = s1 ? 1 : q[2].cy - q[0].cy;
  if (s2 && (q[1].cx - q[0].cx != SH || (SH != 0 && SH != 1))) return false;
  SconvCells c{};
  c.C = q[0].K / (T * T);
  const int smem = sconv_cells_smem(c.C, T);
  if (smem > SL_SMEM) return false;
  c.Wo = q[0].Wo;
  c.HWo = q[0].HWo;
  c.Ho = (int)(c.HWo / c.Wo);
  c.nJ = (c.Wo + 1) / 2;
  c.Pm = (c.Ho + 1) / 2 * c.nJ;
  const long long M = (long long)R * c.Pm;
  if (M <= 0 || M >= (1LL << 31)) return false;
  c.M = (uint32_t)M;
  c.dPm.set(c.Pm);
  c.dnJ.set(c.nJ);
  c.Hs = q[0].Hs;
  c.Ws = q[0].Ws;
  c.HWs = q[0].HWs;
  c.ms = s1 ? 2 : 1;
  c.cy = q[0].cy - (T - 1);
  c.cx = q[0].cx - (T - 1);
  for (int z = 0; z < 4; ++z) c.B[z] = q[s1 ? 0 : z].B;
  const unsigned grid = (unsigned)((M + SL_THREADS * SL_CELLS - 1) / (SL_THREADS * SL_CELLS));
  if (s1) cells_launch<3, 1>(q[0].N, grid, smem, c, src, sstride, out, ostride, s);
  else if (SH) cells_launch<2, 1>(q[0].N, grid, smem, c, src, sstride, out, ostride, s);
  else cells_launch<2, 0>(q[0].N, grid, smem, c, src, sstride, out, ostride, s);
  ++g_launches;
  return true;
}

// The n passes of one contraction (a layer's stride phases, or its forward pass) for R rows.
int sc_launch(const SconvPass* qs, int n, int R, const float* src, long long sstride, float* out, long long ostride,
              const float* bias, cudaStream_t s) {
  if (!bias && cells_try(qs, n, R, src, sstride, out, ostride, s)) return BCROWN_OK;
  for (int i0 = 0; i0 < n; i0 += SC_PHASES) {
    SconvPhases ph{};
    const int nz = std::min(SC_PHASES, n - i0);
    long long M = 0;
    int K = 0;
    for (int z = 0; z < nz; ++z) {
      ph.p[z] = qs[i0 + z];
      const long long m = (long long)R * ph.p[z].Pm;
      if (m >= (1LL << 31)) return fail(BCROWN_ERR_ARG, "FP32 conv: more than 2^31 positions in a chunk");
      ph.p[z].M = (uint32_t)m;
      M = std::max(M, m);
      K = std::max(K, ph.p[z].K);
    }
    if (M <= 0) continue;
    const int N = ph.p[0].N;
    if (N <= 4) {
      const dim3 grid((unsigned)((M + SN_THREADS * SN_TM - 1) / (SN_THREADS * SN_TM)), 1, nz);
      const int smem = sconv_narrow_smem(K);
      if (N == 1) k_sconv_narrow<1><<<grid, SN_THREADS, smem, s>>>(ph, src, sstride, out, ostride, bias);
      else if (N == 2) k_sconv_narrow<2><<<grid, SN_THREADS, smem, s>>>(ph, src, sstride, out, ostride, bias);
      else if (N == 3) k_sconv_narrow<3><<<grid, SN_THREADS, smem, s>>>(ph, src, sstride, out, ostride, bias);
      else k_sconv_narrow<4><<<grid, SN_THREADS, smem, s>>>(ph, src, sstride, out, ostride, bias);
    } else {
      const int BN = N <= 16 ? 16 : N <= 32 ? 32 : N <= 64 ? 64 : 128;
      const dim3 grid((unsigned)((M + SC_BM - 1) / SC_BM), (unsigned)((N + BN - 1) / BN), nz);
      const int smem = sconv_smem(BN, K);
      if (BN == 16) k_sconv<16><<<grid, 32, smem, s>>>(ph, src, sstride, out, ostride, bias);
      else if (BN == 32) k_sconv<32><<<grid, 64, smem, s>>>(ph, src, sstride, out, ostride, bias);
      else if (BN == 64) k_sconv<64><<<grid, 128, smem, s>>>(ph, src, sstride, out, ostride, bias);
      else k_sconv<128><<<grid, 256, smem, s>>>(ph, src, sstride, out, ostride, bias);
    }
    ++g_launches;
  }
  return BCROWN_OK;
}

}  // namespace

bool sconv_supported(const bcrown_net* net, int i) {
  const LayerDev& l = net->ly[i - 1];
  if (l.kind != BCROWN_LAYER_CONV) return false;
  const int T = (l.k + l.stride - 1) / l.stride;
  return (long long)l.out_c * T * T <= SCONV_MAX_K && (long long)l.in_c * l.k * l.k <= SCONV_MAX_K &&
         (long long)l.out_c * l.out_h * l.out_w < (1LL << 31) && (long long)l.in_c * l.in_h * l.in_w < (1LL << 31);
}

int sconv_load(bcrown_net* net) { return sc_prepare(net, sc_of(net)); }

int sconv_bwd(bcrown_net* net, int i, int R, const float* Lam, float* Ain, cudaStream_t s) {
  SconvNet* t = sc_of(net);
  if (!t->ready) return fail(BCROWN_ERR_ARG, "FP32 conv: tables not built");
  const LayerDev& l = net->ly[i - 1];
  const std::vector<SconvPass>& q = t->ly[i].bwd;
  return sc_launch(q.data(), (int)q.size(), R, Lam, l.d_out, Ain, l.d_in, nullptr, s);
}

bool root_patch(const bcrown_net* net, int T, std::vector<int>& n) {
  n.assign(T + 1, 1);
  for (int m = T; m >= 1; --m) {
    const LayerDev& l = net->ly[m - 1];
    if (l.kind != BCROWN_LAYER_CONV || (m < T && !sconv_supported(net, m))) return false;
    const long long nm = (long long)(n[m] - 1) * l.stride + l.k;
    if (nm > 32768 || nm * nm * l.in_c > (long long)l.d_in) return false;
    n[m - 1] = (int)nm;
  }
  return true;
}

int sconv_patch(bcrown_net* net, int T, int i, int R, const float* Lam, float* Ain, cudaStream_t s) {
  SconvNet* t = sc_of(net);
  std::vector<int> n;
  if (!t->ready || !root_patch(net, T, n)) return fail(BCROWN_ERR_ARG, "FP32 conv: no patch tables");
  const LayerDev& l = net->ly[i - 1];
  const std::vector<SconvPass>& q = t->ly[i].patch[T];
  return sc_launch(q.data(), (int)q.size(), R, Lam, (long long)l.out_c * n[i] * n[i], Ain,
                   (long long)l.in_c * n[i - 1] * n[i - 1], nullptr, s);
}

int sconv_fwd(bcrown_net* net, int i, int R, const float* h, float* Z, const float* bias, cudaStream_t s) {
  SconvNet* t = sc_of(net);
  if (!t->ready) return fail(BCROWN_ERR_ARG, "FP32 conv: tables not built");
  const LayerDev& l = net->ly[i - 1];
  return sc_launch(&t->ly[i].fwd, 1, R, h, l.d_in, Z, l.d_out, bias, s);
}

void sconv_release(const bcrown_net* net) {
  std::lock_guard<std::mutex> g(g_sc_mu);
  for (size_t i = 0; i < g_sc.size(); ++i)
    if (g_sc[i].first == net) {
      for (void* b : g_sc[i].second->bufs) cudaFree(b);
      delete g_sc[i].second;
      g_sc.erase(g_sc.begin() + i);
      return;
    }
}

}  // namespace bcrown
