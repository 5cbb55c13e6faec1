// BF16 layer-by-layer bound pass (sm_103a: tcgen05 + TMA) for the networks the fused kernel does
// not take: convolutional networks and fully connected layers wider than 256 neurons.
//
// The recursion of Theorem 3.1 (Eq. definition_A) runs one contraction per launch, and each
// launch's epilogue takes the next step of the recursion on the accumulator it just produced,
// so no FP32 intermediate goes through HBM:
//
//   backward, layer i:  A^(i-1) = Lambda^(i) W^(i)   (a transposed convolution: one GEMM per
//                       stride phase; a fully connected layer: one GEMM)
//                       epilogue: the relaxation of layer i-1 (Lemma 2.1 / Eq. definition_D with
//                       split overriding stability), Lambda^(i-1) = A D + beta S, the bias sums
//                       c += Lambda b + A lambda, and Lambda^(i-1) stored in BF16 as the next
//                       GEMM's operand; for i = 1 the concretisation over the box (Eq.
//                       beta_crown_lp) and x* (x_lo where A^(0) >= 0, else x_hi).
//   forward (adjoint), layer i:  zhat^(i) = W^(i) h^(i-1) + b^(i)
//                       epilogue: dalpha = A zhat (unstable, unsplit, A >= 0), dbeta = S zhat,
//                       h^(i) = D zhat + lambda stored in BF16 as the next operand.
//
// Activations are BF16 in NHWC order (channels innermost, padded to a multiple of 8).  The GEMM
// operand -- rows = (subdomain row, output position), K = (tap, channel) -- comes by TMA where an M
// tile is one box of the map, else it is gathered into shared memory in 16-byte pieces of 8 channels
// by gather warps, one per stage of the ring (at most 4).  TMA streams the weights, one warp issues
// the MMAs into up to four TMEM accumulators (two for 256-column tiles), and as many groups of 4
// epilogue warps read them, each group its own, so that their tiles' epilogues run at once.
// The bias sums of each row are written as partial sums (one slot per position block and column
// group) and added in a fixed order at the end, so the result does not depend on scheduling.
// A at the unstable neurons is stashed in BF16, laid out like alpha, for the adjoint pass; its
// sign is kept even where it rounds to zero, so both passes take the same relaxation branch.
//
// Every mbarrier wait is bounded; on expiry the kernel records BCROWN_ERR_TIMEOUT, raises its
// abort flag, waits (bounded) for its copies in flight, frees TMEM and returns.
#include <algorithm>
#include <atomic>
#include <mutex>
#include <vector>

#include "layer_ring.h"
#include "layer_tc.cuh"
#include "tc_ptx.cuh"

namespace bcrown {

extern std::atomic<long long> g_launches;

namespace lt {

using namespace tc;

// An epilogue warp's list of special elements (32 lanes x at most 16 columns, or 64 columns that hold
// fewer) and its lanes' rows.
constexpr int CAP = 512;
struct LtList {
  int4 row[32][2];           // {alpha base lo, hi, neuron table offset lo, hi}, {output offset lo, hi, chord base lo, hi}
  float val[CAP];
  uint16_t ent[CAP];         // column | lane << 8 | split << 15
  // the splits of the warp's row in this layer, where its positions lie in one row of a convolution
  // (at most 256 channels, 2^22 positions): packed entry, channel | position << 9
  int2 split[BCROWN_MAX_SPLITS];
};

// Warp roles.  Gathered A operand: 12 epilogue warps (three groups of 4, every third tile) and 4
// gather warps.  A operand by TMA: 16 epilogue warps (four groups).  Both with
// the TMA and the MMA warp: 18 warps, which leaves 96 registers a thread.
template <bool TA>
struct LtRoles {
  static constexpr int EPI = TA ? 16 : 12;   // epilogue warps
  static constexpr int NGRP = EPI / 4;       // epilogue groups, one TMEM accumulator each
  static constexpr int GW = TA ? 0 : NS_GATHER;   // gather warps
  static constexpr int TMA_W = EPI, MMA_W = EPI + 1, GATHER0 = EPI + 2;
  static constexpr int THREADS = (EPI + 2 + GW) * 32;
};
constexpr int MAX_NP = 256;
constexpr int MAX_KP = 2048;

enum { EPI_RELAX = 0, EPI_CONCRETIZE = 1, EPI_FWD = 2 };

// One GEMM launch: M = (row, position of this pass) pairs, N = output channels (or, for a fully
// connected pass over a map, NHWC output indices), K = (tap, input channel).
struct Pass {
  long long M;
  int Pm, nJ;                // positions per row in this pass; the pass grid's width
  int N, Np, ntn, nkb, brow; // N in ntn tiles of Np; K blocks; first row of the B matrix in its map
  // gather source: NHWC BF16 map, row stride src_stride elements; the base position of
  // (row, pp = i * nJ + j) is (i * ms + cy, j * ms + cx); table entries per 8-channel chunk of K
  const __nv_bfloat16* src;
  long long src_stride;
  int Hs, Ws, Cps, ms, cy, cx, kchunks;
  const int2* tab;           // [kchunks]: {element offset, dy & 0xffff | dx << 16}; null: chunk
                             // kc is elements 8 kc .. 8 kc + 7 of the row (fully connected)
  // output position of (row, pp): (oa + os * i) * Wo + ob + os * j; npos: position from n
  int oa, ob, os, Wo, npos;
  int Co, HWo, Cpo;          // output map: channels, positions, padded channels
  FastDiv dPm, dnJ, dntn, dHWo;   // (set at the launch)
  __nv_bfloat16* dst;        // NHWC BF16 output (null: none)
  long long dst_stride;
  int layer;                 // hidden layer of the epilogue (0: the input)
  const float* bnhwc;        // its bias in NHWC order (padded channels 0)
  const uint32_t* ntab;      // its neurons in NHWC order, property 0 (stride Ctx::NH per property):
                             // code (0 inactive, 1 active, 2 unstable) | rank among the unstable << 2
  const uint16_t* mtab;      // the same per 8 neurons (stride NH / 8): active bits | unstable bits << 8
  int slot0;                 // first partial-sum slot of this pass
  // A operand by TMA instead of the gather warps: 0 gathered; 4: one box [64 channels][bw][bh][br]
  // of the NHWC source per (tap, 64-channel block) -- an M tile is br rows x bh x bw positions;
  // 2: one box [64][128 rows] of a fully connected pass's linear source; 8: a source of 8 (padded)
  // channels, one unswizzled box [8][bw][bh][br] per tap, 8 taps per K block
  int ta = 0, bw = 0, bh = 0, br = 0;
  const int4* ktab = nullptr;   // ta == 4: per K block {first channel, dy, dx, tap in use};
                                // ta == 8: the same per tap (8 per K block)
};

// Per-call context of the epilogues.
struct Ctx {
  int r0, R, K, P, H, d0, S;
  FastDiv dK;
  BatchView bt;
  Tables tb;
  const float* x_lo;
  const float* x_hi;
  const float* alpha;
  const float* beta;
  int64_t n_alpha, n_beta;
  float* dalpha;
  float* dbeta;
  __nv_bfloat16* stash;      // A at the unstable neurons (alpha layout), or null
  float* cpart;              // [R][S] partial sums of c
  int* status;
  // built once per call by k_lt_rows (rows indexed from 0 = the call's first row)
  const int4* rowinfo;       // [B*K]: {abase lo, abase hi, bbase, prop | valid << 31}
  const uint32_t* ssplit;    // [B][64]: a subdomain's splits sorted by layer, j | t << 20 | (S = +1) << 26
  const int* slayer;         // [B][L + 1]: start of layer l's entries in the subdomain's sorted list
  int L;
  long long NH;              // entries per property in the NHWC neuron table (all hidden layers)
  const float2* chord;       // [P][H]: upper chord (slope, intercept) of the property's unstable
                             // neuron of each rank
};

// Packed split entry of the sorted lists (neuron index j < 2^20, list position t < 64).
__device__ __forceinline__ int sp_j(uint32_t e) { return (int)(e & 0xFFFFFu); }
__device__ __forceinline__ int sp_t(uint32_t e) { return (int)((e >> 20) & 63u); }
__device__ __forceinline__ int sp_s(uint32_t e) { return (e >> 26) & 1u ? 1 : -1; }

__device__ __forceinline__ bool lt_wait(uint64_t* b, uint32_t parity, volatile int* abort, int* status) {
  if (mbar_try(b, parity)) return true;
  long long t0 = clock64();
  while (true) {
    if (mbar_try_sleep(b, parity, 20000u)) return true;
    if (*abort) return false;
    if (clock64() - t0 > 4000000000LL) {
      atomicCAS(status, 0, BCROWN_ERR_TIMEOUT);
      *abort = 1;
      return false;
    }
  }
}

// The TMA and the MMA warp wait with all lanes.
__device__ __forceinline__ bool lt_wait_all(uint64_t* b, uint32_t parity, volatile int* abort, int* status) {
  return mbar_wait_together(b, parity, [&] { return *abort != 0; },
                            [&] {
                              atomicCAS(status, 0, BCROWN_ERR_TIMEOUT);
                              *abort = 1;
                            });
}

__device__ __forceinline__ uint4 ldg_nc_v4(const void* p, bool pred) {
  uint4 v;
  asm volatile(
      "{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %5, 0;\n\tmov.b32 %0, 0;\n\tmov.b32 %1, 0;\n\tmov.b32 %2, 0;\n\t"
      "mov.b32 %3, 0;\n\t@q ld.global.nc.v4.b32 {%0, %1, %2, %3}, [%4];\n\t}"
      : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
      : "l"(p), "r"((uint32_t)pred)
      : "memory");
  return v;
}

// BF16 of a, rounded to nearest, keeping a < 0 negative (the smallest negative subnormal where it
// would round to -0), so a sign test on the stash agrees with the one on a.
__device__ __forceinline__ __nv_bfloat16 bf16_signed(float a) {
  __nv_bfloat16 h = __float2bfloat16_rn(a);
  if (a < 0.f && !(__bfloat162float(h) < 0.f)) h = __ushort_as_bfloat16((unsigned short)0x8001u);
  return h;
}

__device__ __forceinline__ uint32_t pack2(float lo, float hi) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&v);
}

__device__ __forceinline__ float lt_warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

template <int MODE, bool TA>
__global__ void __launch_bounds__(LtRoles<TA>::THREADS, 1)
    k_lt(const __grid_constant__ CUtensorMap mapB, const __grid_constant__ CUtensorMap mapA, const Pass ps,
         const Ctx cx) {
  using RL = LtRoles<TA>;
  const long long M = ps.M;
  const int Np = ps.Np, nkb = ps.nkb;
  extern __shared__ __align__(1024) uint8_t lsm_raw[];
  const uint32_t pad = (1024u - (su32(lsm_raw) & 1023u)) & 1023u;
  uint8_t* base = lsm_raw + pad;
  const int bbytes = Np * 128;
  const int NS = lt_stages(TA, Np);
  uint8_t* sA = base;                                  // NS x 16 KB
  uint8_t* sB = base + NS * 16384;                     // NS x Np * 128
  uint64_t* bars = reinterpret_cast<uint64_t*>(sB + NS * bbytes);
  uint64_t* full = bars;
  uint64_t* empty = bars + NS_MAX;
  uint64_t* acc_full = bars + 2 * NS_MAX;    // up to 4 accumulators
  uint64_t* acc_empty = bars + 2 * NS_MAX + 4;
  uint32_t* tbase_sm = reinterpret_cast<uint32_t*>(bars + 2 * NS_MAX + 8);
  volatile int* abort = reinterpret_cast<volatile int*>(tbase_sm + 1);
  int2* stab = reinterpret_cast<int2*>(bars + 32);     // 256 bytes past the barriers
  float* sbias = reinterpret_cast<float*>(stab + MAX_KP / 8);   // conv passes: the layer's channel biases
  LtList* slist = reinterpret_cast<LtList*>(sbias + MAX_NP);    // one per epilogue warp
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const long long ntiles = (M + 127) / 128 * ps.ntn;   // tile = m tile * ntn + n tile
  // accumulators in use: one per epilogue group, as many groups as their Np columns each fit in
  // TMEM's 512 (the other groups then idle)
  const int ngrp = RL::NGRP * Np <= 512 ? RL::NGRP : (3 * Np <= 512 ? min(3, RL::NGRP) : 2);
  const uint32_t need = (uint32_t)(ngrp * Np);
  const uint32_t tcols = need <= 32 ? 32u : (need <= 64 ? 64u : (need <= 128 ? 128u : (need <= 256 ? 256u : 512u)));
  if (threadIdx.x == 0) {
    for (int i = 0; i < NS; ++i) {
      mbar_init(&full[i], TA ? 1 : 2);   // the TMA transaction (and the stage's gather warp)
      mbar_init(&empty[i], 1);
    }
    for (int i = 0; i < RL::NGRP; ++i) {
      mbar_init(&acc_full[i], 1);
      mbar_init(&acc_empty[i], 4);   // the 4 warps of the epilogue group of buffer i
    }
    *abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == RL::MMA_W) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(tbase_sm)), "r"(tcols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tbase_sm;

  if (warp == RL::TMA_W) {
    // ------------------------------------------------------------ weights (B) by TMA, and A with TA
    // The whole warp runs the loop and one elected lane issues: no division and no global load per
    // K block (the tile's coordinates are worked out once per tile, the tap table is in shared
    // memory, the gathering kernel's table space).
    int4* sktab = reinterpret_cast<int4*>(stab);
    if (TA && (ps.ta == 4 || ps.ta == 8)) {
      for (int k = lane; k < (ps.ta == 8 ? 8 * nkb : nkb); k += 32) sktab[k] = ps.ktab[k];
      __syncwarp();
    }
    uint32_t seq = 0;
    int st = 0;
    uint32_t ph = 0;   // parity of the current pass over the ring
    bool ok = true;
    for (long long tile = blockIdx.x; tile < ntiles && ok; tile += gridDim.x) {
      const long long mt = tile / ps.ntn;
      const int brow = ps.brow + (int)(tile - mt * ps.ntn) * Np;
      int ax = 0, ay = 0, ar = 0;   // TA: the box origin of the tile's first position, tap 0
      if constexpr (TA) {
        const long long m0 = mt * 128;
        if (ps.ta == 2) {
          ar = (int)m0;
        } else {
          const long long r0 = m0 / ps.Pm;
          const int pp0 = (int)(m0 - r0 * ps.Pm);
          const int i0 = pp0 / ps.nJ;
          ax = (pp0 - i0 * ps.nJ) * ps.ms + ps.cx;
          ay = i0 * ps.ms + ps.cy;
          ar = (int)r0;
        }
      }
      for (int kb = 0; kb < nkb; ++kb, ++seq) {
        if (!lt_wait_all(&empty[st], ph ^ 1, abort, cx.status)) {
          ok = false;
          break;
        }
        if (lane == 0) {
          mbar_expect_tx(&full[st], (TA ? 16384u : 0u) + (uint32_t)bbytes);
          if constexpr (TA) {
            if (ps.ta == 2) {
              tma_load_2d(sA + st * 16384, &mapA, kb * 64, ar, &full[st]);
            } else if (ps.ta == 8) {
              // 8 channels per tap: the K block is 8 taps, one box of 16-byte rows each, 2 KB apart
#pragma unroll 1
              for (int j = 0; j < 8; ++j) {
                const int4 kt = sktab[kb * 8 + j];
                const int y = kt.w ? ay + kt.y : -(1 << 20);
                tma_load_4d(sA + st * 16384 + j * 2048, &mapA, 0, ax + kt.z, y, ar, &full[st]);
              }
            } else {
              const int4 kt = sktab[kb];
              // a K block past the phase's taps reads a box outside the map: zeros
              const int y = kt.w ? ay + kt.y : -(1 << 20);
              tma_load_4d(sA + st * 16384, &mapA, kt.x, ax + kt.z, y, ar, &full[st]);
            }
          }
          tma_load_2d(sB + st * bbytes, &mapB, kb * 64, brow, &full[st]);
        }
        if (++st == NS) st = 0, ph ^= 1;
      }
    }
    if (!ok && lane == 0) {
      for (uint32_t q = (seq > (uint32_t)NS ? seq - NS : 0); q < seq; ++q) {
        long long t0 = clock64();
        while (!mbar_try(&full[q % NS], (q / NS) & 1) && clock64() - t0 < 200000000LL) {
        }
      }
    }
  } else if (warp == RL::MMA_W) {
    // ------------------------------------------------------------ MMA issuer
    // (whole warp, one elected lane issues: see umma_kpair)
    uint32_t buf = 0, cph = 1, wph = 0;
    int st = 0;
    bool ok = true;
    const uint32_t idesc = idesc_bf16(Np);
    const uint32_t b0 = sdesc_lo(su32(sB)), bstep = (uint32_t)bbytes >> 4;
    const bool plain = TA && ps.ta == 8;   // A without swizzle: core matrices 128 B apart along M, 2 KB along K
    const uint32_t a0 = plain ? sdesc_plain_lo(su32(sA), 2048) : sdesc_lo(su32(sA));
    const uint32_t b_empty = su32(empty), b_acc = su32(acc_full);
    for (long long tile = blockIdx.x; tile < ntiles && ok; tile += gridDim.x) {
      if (!lt_wait_all(&acc_empty[buf], cph, abort, cx.status)) break;
      tc_fence_after();
      const uint32_t dt = tmem + buf * (uint32_t)Np;
      for (int kb = 0; kb < nkb; ++kb) {
        if (!lt_wait_all(&full[st], wph, abort, cx.status)) {
          ok = false;
          break;
        }
        tc_fence_after();
        const uint32_t al = a0 + (uint32_t)st * (16384 >> 4), bl = b0 + (uint32_t)st * bstep;
        if (plain)
          umma_kblock_warp<SDESC_PLAIN_HI(128), (4096 >> 4)>(dt, al, bl, idesc, kb != 0 ? 1u : 0u, b_empty + 8 * st);
        else
          umma_kblock_warp<SDESC_HI, 2>(dt, al, bl, idesc, kb != 0 ? 1u : 0u, b_empty + 8 * st);
        if (++st == NS) st = 0, wph ^= 1;
      }
      if (!ok) break;
      umma_commit_warp(b_acc + 8 * buf);
      if (++buf == (uint32_t)ngrp) buf = 0, cph ^= 1;
    }
  } else if (!TA && warp >= RL::GATHER0) {
    // ------------------------------------------------------------ operand (A) gather
    // warp g takes the K blocks g, g + NS, ... of the (tile, K block) order, all of them in ring slot g
    // (lt_gather_warp); a block is 8 chunks of 16 bytes per row
    const int g = warp - RL::GATHER0;
    constexpr int GW = RL::GW > 0 ? RL::GW : 1;
    const bool linear = ps.tab == nullptr;
    if (!linear)
      for (int k = threadIdx.x - RL::GATHER0 * 32; k < ps.kchunks; k += GW * 32) stab[k] = ps.tab[k];
    asm volatile("bar.sync 2, %0;" ::"n"(GW * 32) : "memory");
    int next = 0;       // stage of the next block, and the parity of its empty barrier
    uint32_t par = 1;
    bool ok = true;
    for (long long tile = blockIdx.x; tile < ntiles && ok; tile += gridDim.x) {
      const __nv_bfloat16* srow[4];
      int y0[4], x0[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const long long m = tile / ps.ntn * 128 + lane + 32 * q;
        const bool mv = m < M;
        const long long r = mv ? m / ps.Pm : 0;
        const int pp = mv ? (int)(m - r * ps.Pm) : 0;
        const int i = pp / ps.nJ, j = pp - (pp / ps.nJ) * ps.nJ;
        y0[q] = mv ? i * ps.ms + ps.cy : -32768;
        x0[q] = j * ps.ms + ps.cx;
        srow[q] = ps.src + r * ps.src_stride + (mv ? ((long long)y0[q] * ps.Ws + x0[q]) * ps.Cps : 0);
      }
      for (int kb = 0; kb < nkb; ++kb) {
        const bool mine = lt_gather_warp(next) == g;
        const uint32_t ph = par;
        if (++next == NS) next = 0, par ^= 1;
        if (!mine) continue;
        int okw = 1;
        if (lane == 0) okw = lt_wait(&empty[g], ph, abort, cx.status) ? 1 : 0;
        okw = __shfl_sync(0xffffffffu, okw, 0);
        if (!okw) {
          ok = false;
          break;
        }
        uint8_t* stage = sA + g * 16384;
        // 4 chunks (of 4 rows each) in flight at a time: 16 loads of 16 bytes per lane
#pragma unroll
        for (int c0 = 0; c0 < 8; c0 += 4) {
          uint4 v[4][4];
#pragma unroll
          for (int cc = 0; cc < 4; ++cc) {
            const int kc = kb * 8 + c0 + cc;
            const int2 t = kc < ps.kchunks ? (linear ? make_int2(8 * kc, 0) : stab[kc]) : make_int2(0, 0x8000);
            const int dy = (int)(short)(t.y & 0xffff), dx = t.y >> 16;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              const bool in = (unsigned)(y0[q] + dy) < (unsigned)ps.Hs && (unsigned)(x0[q] + dx) < (unsigned)ps.Ws;
              v[cc][q] = ldg_nc_v4(srow[q] + t.x, in);
            }
          }
#pragma unroll
          for (int cc = 0; cc < 4; ++cc) {
            const int c = c0 + cc;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              const int m = lane + 32 * q;
              *reinterpret_cast<uint4*>(stage + m * 128 + ((c ^ (m & 7)) << 4)) = v[cc][q];
            }
          }
        }
        fence_proxy_async();   // generic-proxy stores of the stage, before the MMA reads it
        __syncwarp();
        if (lane == 0) mbar_arrive(&full[g]);
      }
    }
  } else {
    // ------------------------------------------------------------ epilogue
    // ngrp groups of 4 warps take every ngrp-th tile (group g: accumulator buffer g), so that
    // their tiles' epilogues overlap; warp w of a group reads TMEM lanes 32 (w % 4) .. + 31 (M
    // rows) and every column chunk of 8
    const int q4 = warp & 3, eg = warp >> 2;
    uint32_t accseq = eg;   // this group takes the CTA's tiles eg, eg + ngrp, ...
    const bool sb_smem = MODE != EPI_CONCRETIZE && !ps.npos && ps.Cpo <= MAX_NP;
    if (sb_smem) {
      // a conv layer's bias is per channel: bnhwc at position 0
      for (int c = threadIdx.x; c < MAX_NP; c += RL::EPI * 32) sbias[c] = c < ps.Cpo ? ps.bnhwc[c] : 0.f;
      asm volatile("bar.sync 1, %0;" ::"n"(RL::EPI * 32) : "memory");
    }
    const bool warp_sum_ok = (ps.Pm & 31) == 0;   // 32 lanes = 32 positions of one row
    for (long long tile = blockIdx.x + (long long)eg * gridDim.x; eg < ngrp && tile < ntiles;
         tile += (long long)ngrp * gridDim.x, accseq += ngrp) {
      const int buf = eg;
      // (fewer than 2^31 positions a launch: the rows of a chunk are bounded by its 16 GB)
      const uint32_t mt = ps.dntn((uint32_t)tile);
      const int nt = (int)((uint32_t)tile - mt * ps.dntn.d);
      const uint32_t m = mt * 128 + 32 * q4 + lane;
      const bool mv = m < (uint32_t)M;
      const int rl = mv ? (int)ps.dPm(m) : 0;                 // row within the chunk
      const int pp = mv ? (int)(m - (uint32_t)rl * ps.dPm.d) : 0;
      const int pi = (int)ps.dnJ((uint32_t)pp), pj = pp - pi * ps.nJ;
      const int pm = ps.npos ? 0 : (ps.oa + ps.os * pi) * ps.Wo + ps.ob + ps.os * pj;
      // the row: subdomain b, spec k, property p (one 16-byte load of the row table)
      const int r = cx.r0 + rl;
      const int b = (int)cx.dK((uint32_t)r);
      const int4 ri = mv ? cx.rowinfo[r] : make_int4(0, 0, 0, 0);
      int s0 = 0, s1 = 0;
      if (mv && MODE != EPI_CONCRETIZE) {
        const int* sl = cx.slayer + (size_t)b * (cx.L + 1) + ps.layer;
        s0 = b * BCROWN_MAX_SPLITS + sl[0];
        s1 = b * BCROWN_MAX_SPLITS + sl[1];
      }
      const long long abase = ((long long)(uint32_t)ri.y << 32) | (uint32_t)ri.x;
      const long long bbase = ri.z;
      const int prop = ri.w & 0x7FFFFFFF;
      const bool rv = mv && (ri.w < 0);
      const int nlo = nt * Np;
      // the row's splits in this layer: element n and position of an entry (n: the NHWC index of a
      // fully connected pass over a map, whose one position stands for all)
      auto place = [&](uint32_t e, int& n, int& p) {
        const int jn = sp_j(e);
        const int c = (int)ps.dHWo((uint32_t)jn);
        p = jn - c * ps.HWo;
        n = c;
        if (ps.npos) n += p * ps.Cpo, p = 0;
      };
      const int pos_here = ps.npos ? 0 : pm;
      int nsplit = 0;
      if constexpr (MODE != EPI_CONCRETIZE) {
        nsplit = rv ? s1 - s0 : 0;
        __syncwarp();
        if (warp_sum_ok) {   // one row per warp: the lanes place its entries once, for all
          nsplit = __shfl_sync(0xffffffffu, nsplit, 0);
          const int f = __shfl_sync(0xffffffffu, s0, 0);
          for (int q = lane; q < nsplit; q += 32) {
            const uint32_t e = cx.ssplit[f + q];
            int n, p;
            place(e, n, p);
            slist[warp].split[q] = make_int2((int)e, n | p << 9);
          }
        }
      }
      // entry q of this thread's row
      auto split_at = [&](int q, int& n, int& p) -> uint32_t {
        if (warp_sum_ok) {
          const int2 x = slist[warp].split[q];
          n = x.y & 511;
          p = (int)((uint32_t)x.y >> 9);
          return (uint32_t)x.x;
        }
        const uint32_t e = cx.ssplit[s0 + q];
        place(e, n, p);
        return e;
      };
      int okw = 1;
      if constexpr (MODE == EPI_CONCRETIZE) {
        if (lane == 0) okw = lt_wait(&acc_full[buf], (accseq / (uint32_t)ngrp) & 1, abort, cx.status) ? 1 : 0;
        okw = __shfl_sync(0xffffffffu, okw, 0);
        if (!okw) break;
        tc_fence_after();
      }
      float acc = 0.f, acc_special = 0.f;
      const uint32_t tacc = tmem + ((uint32_t)(32 * q4) << 16) + (uint32_t)(buf * Np);
      __nv_bfloat16* dst_r = ps.dst ? ps.dst + (long long)rl * ps.dst_stride : nullptr;
      // the NHWC index of element n of this thread's position (fully connected over a map: n itself)
      const long long nhwc0 = ps.npos ? 0 : (long long)pm * ps.Cpo;
      if constexpr (MODE == EPI_CONCRETIZE) {
        for (int n0 = 0; n0 < Np; n0 += 8) {
          float v[8];
          tmem_ld8(tacc + n0, v);
          const int nb = nlo + n0;   // first n of the chunk
          if (mv && nb < ps.N) {
            float o[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) {
              const int n = nb + e;
              o[e] = 0.f;
              if (!rv || n >= ps.Co) continue;
              const int jl = n * ps.HWo + pm;   // input coordinate (channel-major)
              const float a = v[e];
              const float xl = cx.x_lo[(size_t)prop * cx.d0 + jl], xh = cx.x_hi[(size_t)prop * cx.d0 + jl];
              acc += fminf(a * xl, a * xh);
              o[e] = a >= 0.f ? xl : xh;   // x* minimises A^(0) x over the box
            }
            if (dst_r && nb + 8 <= (ps.npos ? ps.N : ps.Cpo))
              *reinterpret_cast<uint4*>(dst_r + nhwc0 + nb) =
                  make_uint4(pack2(o[0], o[1]), pack2(o[2], o[3]), pack2(o[4], o[5]), pack2(o[6], o[7]));
          }
        }
      } else {
        // Most neurons are stable and unsplit and need no load of their own: 8 columns at a time
        // they take D = 1 or 0 from bit masks.  The special ones (unstable or split; 5 to 35 % on the
        // convolutional maps) leave their value in the warp's list, whose entries the 32 lanes then
        // share out evenly, 4 each at a time, whichever position they lie at; each overwrites its
        // element of the output.  The list's order is known from the masks before the accumulator is
        // complete, so the first 4 entries' ranks are loaded during that wait and their alpha, chord
        // and stash during the pass over the columns: what bounds this kernel is the latency of
        // those dependent loads.  A split element is worked off by its own lane.  Measured on the
        // CIFAR-shaped 4-conv network at 9,216 rows, bound and gradient: 14.2 ms with one pass over
        // all elements, the special ones' loads predicated (71 instructions an element); 14.8 with a
        // list per lane, which waits for the longest one's loads; 8.7 with this.
        LtList& wl = slist[warp];
        const long long tofs = (long long)prop * cx.NH + nhwc0;   // the position's neurons in the tables
        const int lim = ps.npos ? ps.N : ps.Cpo;                  // elements that exist in the map
        __syncwarp();
        {
          const long long dofs = (long long)rl * ps.dst_stride + nhwc0, cofs = (long long)prop * cx.H;
          wl.row[lane][0] = make_int4(ri.x, ri.y, (int)(uint32_t)tofs, (int)(tofs >> 32));
          wl.row[lane][1] = make_int4((int)(uint32_t)dofs, (int)(dofs >> 32), (int)(uint32_t)cofs, (int)(cofs >> 32));
        }
        const bool mvec = ((ps.Cpo | ps.N) & 63) == 0 && !(nlo & 63);   // 64 columns' masks in one 16-byte load
        bool waited = false;
        for (int cb = 0; cb < Np && okw; cb += 64) {
          const int nb0 = nlo + cb, wid = min(64, Np - cb);
          // the block's active and unstable bits
          uint32_t w[4] = {0u, 0u, 0u, 0u};
          if (rv && mvec && nb0 < lim) {
            const uint4 x = *reinterpret_cast<const uint4*>(ps.mtab + (tofs + nb0) / 8);
            w[0] = x.x, w[1] = x.y, w[2] = x.z, w[3] = x.w;
          } else if (rv) {
#pragma unroll
            for (int c = 0; c < 8; ++c)
              if (8 * c < wid && nb0 + 8 * c < lim)
                w[c >> 1] |= (uint32_t)ps.mtab[(tofs + nb0) / 8 + c] << (16 * (c & 1));
          }
          const unsigned long long act64 =
              (unsigned long long)__byte_perm(w[2], w[3], 0x6420) << 32 | __byte_perm(w[0], w[1], 0x6420);
          unsigned long long spec64 =
              (unsigned long long)__byte_perm(w[2], w[3], 0x7531) << 32 | __byte_perm(w[0], w[1], 0x7531);
          unsigned long long split64 = 0;
          for (int q = 0; q < nsplit; ++q) {
            int n, p;
            split_at(q, n, p);
            if (rv && p == pos_here && (unsigned)(n - nb0) < (unsigned)wid) split64 |= 1ull << (n - nb0);
          }
          spec64 |= split64;
          // 64 columns at once where the list holds their special elements, else 16 at a time
          const int all = __reduce_add_sync(0xffffffffu, __popcll(spec64));
          const int sub = all <= CAP ? wid : 16;
          for (int c0 = 0; c0 < wid && okw; c0 += sub) {
            const unsigned long long range = (sub == 64 ? ~0ull : ((1ull << sub) - 1ull)) << c0;
            unsigned long long spec = spec64 & range;
            const int mine = __popcll(spec);
            int off = mine;   // exclusive prefix over the lanes
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
              const int y = __shfl_up_sync(0xffffffffu, off, o);
              if (lane >= o) off += y;
            }
            const int total = __shfl_sync(0xffffffffu, off, 31);
            off -= mine;
            __syncwarp();   // the list's last use
            for (int i = off; spec; ++i) {
              const int bit = __ffsll((long long)spec) - 1;
              wl.ent[i] = (uint16_t)((cb + bit) | lane << 8 | ((split64 >> bit) & 1ull ? 0x8000 : 0));
              spec &= spec - 1;
            }
            __syncwarp();
            // entries first + lane + 32 q: their ranks (-1: none, or a split one), then alpha and stash.
            // (The rows' bases are read from the list again where they are needed: values that live
            // through the pass over the columns are spilled, and a spilled value's reload misses the
            // little L1 that the stages leave.)
            int rk[4];
            auto ranks = [&](int first) {
#pragma unroll
              for (int q = 0; q < 4; ++q) {
                const int i = first + lane + 32 * q;
                const int en = i < total ? (int)wl.ent[i] : 0x8000;
                rk[q] = -1;
                if (!(en & 0x8000)) {
                  const int4 x = wl.row[en >> 8][0];
                  const long long t = ((long long)x.w << 32) | (uint32_t)x.z;
                  rk[q] = (int)(ps.ntab[t + nlo + (en & 255)] >> 2);
                }
              }
            };
            float al[4];
            uint32_t st[4];
            auto operands = [&](int first) {
#pragma unroll
              for (int q = 0; q < 4; ++q) {
                al[q] = 0.f;
                st[q] = 0u;
                if (rk[q] < 0) continue;
                const int4 x = wl.row[wl.ent[first + lane + 32 * q] >> 8][0];
                const long long ab = (((long long)x.y << 32) | (uint32_t)x.x) + rk[q];
                al[q] = cx.alpha[ab];
                if (MODE == EPI_FWD) st[q] = reinterpret_cast<const uint16_t*>(cx.stash)[ab];
              }
            };
            ranks(0);
            if (!waited) {
              if (lane == 0) okw = lt_wait(&acc_full[buf], (accseq / (uint32_t)ngrp) & 1, abort, cx.status) ? 1 : 0;
              okw = __shfl_sync(0xffffffffu, okw, 0);
              if (!okw) break;
              tc_fence_after();
              waited = true;
            }
            uint32_t u[8];
            __syncwarp();
            tmem_ld8_issue(tacc + cb + c0, u);
            operands(0);
            // the columns
            int put = off;
            unsigned long long actr = act64 >> c0, specr = spec64 >> c0;
#pragma unroll 1
            for (int n0 = cb + c0; n0 < cb + c0 + sub; n0 += 8) {
              const int nb = nlo + n0;   // first n of the chunk
              float v[8];
              __syncwarp();
              tmem_wait8(u);
#pragma unroll
              for (int e = 0; e < 8; ++e) v[e] = __uint_as_float(u[e]);
              if (n0 + 8 < cb + c0 + sub) tmem_ld8_issue(tacc + n0 + 8, u);
              // biases: a conv layer's are per channel (shared memory, up to MAX_NP channels); a fully
              // connected pass's per n, and a wider layer's channels from global memory
              float4 bx = make_float4(0.f, 0.f, 0.f, 0.f), by = bx;
              if (sb_smem) {
                bx = *reinterpret_cast<const float4*>(sbias + nb);
                by = *reinterpret_cast<const float4*>(sbias + nb + 4);
              } else if (nb < lim) {
                bx = *reinterpret_cast<const float4*>(ps.bnhwc + nb);
                by = *reinterpret_cast<const float4*>(ps.bnhwc + nb + 4);
              }
              const float bv[8] = {bx.x, bx.y, bx.z, bx.w, by.x, by.y, by.z, by.w};
              const uint32_t sp8 = (uint32_t)specr & 255u, ac8 = (uint32_t)actr & ~sp8;
              actr >>= 8;
              specr >>= 8;
              float o[8];
#pragma unroll
              for (int e = 0; e < 8; ++e) {
                if (MODE == EPI_RELAX) {
                  o[e] = (ac8 >> e) & 1u ? v[e] : v[e] * 0.f;   // (0, or NaN where A is not finite)
                  acc = fmaf(o[e], bv[e], acc);
                } else {
                  v[e] += bv[e];
                  o[e] = (ac8 >> e) & 1u ? v[e] : 0.f;
                }
                if ((sp8 >> e) & 1u) wl.val[put++] = v[e];
              }
              if (dst_r && mv && nb + 8 <= lim)
                // the chunk's elements are contiguous in the NHWC output
                *reinterpret_cast<uint4*>(dst_r + nhwc0 + nb) = make_uint4(
                    rv ? pack2(o[0], o[1]) : 0u, rv ? pack2(o[2], o[3]) : 0u, rv ? pack2(o[4], o[5]) : 0u,
                    rv ? pack2(o[6], o[7]) : 0u);
            }
            if (cb + c0 + sub == Np) {   // the accumulator has been read: the next tile may take it
              tc_fence_before();
              __syncwarp();
              if (lane == 0) mbar_arrive(&acc_empty[buf]);
            }
            __syncwarp();
            // the special elements, shared out over the lanes
#pragma unroll 1
            for (int first = 0; first < total; first += 128) {
              if (first > 0) {
                ranks(first);
                operands(first);
              }
              float2 ch[4];
#pragma unroll
              for (int q = 0; q < 4; ++q) {
                ch[q] = make_float2(0.f, 0.f);
                if (rk[q] < 0) continue;
                const int4 x = wl.row[wl.ent[first + lane + 32 * q] >> 8][1];
                ch[q] = cx.chord[(((long long)x.w << 32) | (uint32_t)x.z) + rk[q]];
              }
#pragma unroll
              for (int q = 0; q < 4; ++q) {
                if (rk[q] < 0) continue;
                const int i = first + lane + 32 * q, en = wl.ent[i], n = nlo + (en & 255);
                const float a = wl.val[i];
                const int4 rw = wl.row[en >> 8][0];
                const long long ab = (((long long)rw.y << 32) | (uint32_t)rw.x) + rk[q];
                float out;
                if (MODE == EPI_RELAX) {
                  const float bn = sb_smem ? sbias[n] : ps.bnhwc[n];
                  const bool pos = a >= 0.f;
                  const float D = pos ? __saturatef(al[q]) : ch[q].x, lm = pos ? 0.f : ch[q].y;
                  if (cx.stash) cx.stash[ab] = bf16_signed(a);
                  out = a * D;
                  const float c = fmaf(out, bn, a * lm);
                  if (warp_sum_ok) acc += c;   // every lane's position lies in the same row
                  else wl.val[i] = c;
                } else {   // a holds zhat
                  const float A = __uint_as_float(st[q] << 16);
                  const bool pos = A >= 0.f;
                  out = pos ? __saturatef(al[q]) * a : fmaf(ch[q].x, a, ch[q].y);
                  cx.dalpha[ab] = pos ? A * a : 0.f;
                }
                if (ps.dst) {
                  const int4 x = wl.row[en >> 8][1];
                  const long long t = ((long long)x.y << 32) | (uint32_t)x.x;
                  ps.dst[t + n] = __float2bfloat16_rn(out);
                }
              }
            }
            // split elements: rare, by their own lane
            unsigned long long todo = split64 & range;
            while (todo) {
              const int bit = __ffsll((long long)todo) - 1;
              todo &= todo - 1;
              const int n = nb0 + bit;
              const int at = off + __popcll(spec64 & range & ((1ull << bit) - 1ull));
              const float a = wl.val[at];
              const uint32_t ent = ps.ntab[tofs + n];
              const int code = (int)(ent & 3u), rank = (int)(ent >> 2);
              int s = 0, ts = 0;   // its sign and list position (the last entry, as everywhere)
              for (int q = 0; q < nsplit; ++q) {
                int n2, p2;
                const uint32_t e = split_at(q, n2, p2);
                if (p2 == pos_here && n2 == n) {
                  s = sp_s(e);
                  ts = sp_t(e);
                }
              }
              const long long bi = bbase + ts;
              if (bi >= cx.n_beta) atomicCAS(cx.status, 0, BCROWN_ERR_ARG);
              float out;
              if (MODE == EPI_RELAX) {
                const float bn = sb_smem ? sbias[n] : ps.bnhwc[n];
                const float bs = bi < cx.n_beta ? fmaxf(cx.beta[bi], 0.f) * (float)s : 0.f;
                out = fmaf(a, s == -1 ? 1.f : 0.f, bs);
                if (warp_sum_ok) acc = fmaf(out, bn, acc);
                else wl.val[at] = out * bn;
              } else {
                if (bi < cx.n_beta) cx.dbeta[bi] = (float)s * a;
                out = s == -1 ? a : 0.f;
                // a split unstable neuron keeps its alpha slot, which the bound does not use
                if (code == CODE_UNSTABLE) cx.dalpha[abase + rank] = 0.f;
              }
              if (dst_r) dst_r[nhwc0 + n] = __float2bfloat16_rn(out);
            }
            if (MODE == EPI_RELAX && !warp_sum_ok) {
              // each lane adds up its own row's terms in column order, apart from the stable columns': how
              // many columns a list holds depends on the rows that share the warp, the sums do not
              __syncwarp();
              const int end = off + __popcll(spec64 & range);
              for (int i = off; i < end; ++i) acc_special += wl.val[i];
            }
          }
        }
        if (!okw) break;
      }
      if (MODE == EPI_CONCRETIZE) {
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&acc_empty[buf]);
      }
      if (MODE != EPI_FWD) {
        // partial sum of c for (row, this thread's positions and columns); a fixed slot each
        if (warp_sum_ok) {
          const float sw = lt_warp_sum(acc);
          if (lane == 0 && mv)
            cx.cpart[(size_t)rl * cx.S + ps.slot0 + ((size_t)nt * ps.Pm + pp) / 32] = sw;
        } else if (mv) {
          cx.cpart[(size_t)rl * cx.S + ps.slot0 + (size_t)nt * ps.Pm + pp] = acc + acc_special;
        }
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == RL::MMA_W) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(tcols) : "memory");
  }
}

// Top of the recursion: A^(L-1) = Wbar_k, relaxed (layer L-1) into Lambda^(L-1) (NHWC BF16), its
// bias sum into slot 0 and A at the unstable neurons into the stash.  One warp per row.
__global__ void __launch_bounds__(256) k_lt_top(Ctx cx, int layer, long long hoff, int Co, int HWo, int Cpo,
                                                const float* __restrict__ Wbar, const float* __restrict__ bias,
                                                __nv_bfloat16* __restrict__ dst, long long dst_stride) {
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rl = blockIdx.x * 8 + w;
  if (rl >= cx.R) return;
  const int r = cx.r0 + rl;
  const int b = r / cx.K, k = r - b * cx.K;
  const int4 ri = cx.rowinfo[r];
  const long long abase = ((long long)(uint32_t)ri.y << 32) | (uint32_t)ri.x;
  const long long bbase = ri.z;
  const int prop = ri.w & 0x7FFFFFFF;
  const bool rv = ri.w < 0;
  const int* sl = cx.slayer + (size_t)b * (cx.L + 1) + layer;
  const int s0 = b * BCROWN_MAX_SPLITS + sl[0], s1 = b * BCROWN_MAX_SPLITS + sl[1];
  const int d = Co * HWo;
  float acc = 0.f;
  const size_t ng0 = (size_t)prop * cx.H + hoff;
  for (int q = lane; q < HWo * Cpo; q += 32) {
    // NHWC index q = p * Cpo + c
    const int p = q / Cpo, c = q - (q / Cpo) * Cpo;
    float L = 0.f;
    if (rv && c < Co) {
      const int jl = c * HWo + p;
      const float a = Wbar[(size_t)k * d + jl];
      int s = 0, ts = 0;
      for (int u = s0; u < s1; ++u) {
        const uint32_t e = cx.ssplit[u];
        if (sp_j(e) == jl) {
          s = sp_s(e);
          ts = sp_t(e);
        }
      }
      float D, lm = 0.f, bs = 0.f;
      const size_t ng = ng0 + jl;
      if (s != 0) {
        D = s == -1 ? 1.f : 0.f;
        const long long bi = bbase + ts;
        if (bi < cx.n_beta) bs = fmaxf(cx.beta[bi], 0.f) * (float)s;
        else atomicCAS(cx.status, 0, BCROWN_ERR_ARG);
      } else {
        const uint8_t code = cx.tb.code[ng];
        if (code == CODE_ACTIVE) D = 1.f;
        else if (code == CODE_INACTIVE) D = 0.f;
        else {
          const int rk = cx.tb.rank[ng];
          if (a >= 0.f) D = __saturatef(cx.alpha[abase + rk]);
          else {
            D = cx.tb.slope[ng];
            lm = cx.tb.icpt[ng];
          }
          if (cx.stash) cx.stash[abase + rk] = bf16_signed(a);
        }
      }
      L = fmaf(a, D, bs);
      acc = fmaf(L, bias[jl], fmaf(a, lm, acc));
    }
    dst[(size_t)rl * dst_stride + q] = __float2bfloat16_rn(L);
  }
  acc = lt_warp_sum(acc);
  if (lane == 0) cx.cpart[(size_t)rl * cx.S] = acc;
}

// Per row (once per call): where its alpha and beta start, its property, and whether its batch
// entries are consistent (otherwise the row is skipped and BCROWN_ERR_ARG recorded).
__global__ void __launch_bounds__(256) k_lt_rowinfo(int R, int K, int P, BatchView bt, const int32_t* __restrict__ U,
                                                    int64_t n_alpha, int4* __restrict__ rowinfo, int* status) {
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= R) return;
  const int b = r / K, k = r - b * K;
  int prop = bt.prop_of[b];
  bool v = prop >= 0 && prop < P;
  if (!v) prop = 0;
  const int cnt = bt.split_cnt[b], off = bt.split_off[b];
  const int Up = U[prop];
  const long long abase = bt.alpha_off[b] + (long long)k * Up;
  const long long bbase = (long long)off * K + (long long)k * cnt;
  v = v && cnt >= 0 && cnt <= BCROWN_MAX_SPLITS && off >= 0 && abase >= 0 && abase + Up <= n_alpha &&
      bbase <= 0x7FFFFFFFLL;
  if (!v) atomicCAS(status, 0, BCROWN_ERR_ARG);
  rowinfo[r] = make_int4((int)(uint32_t)(abase & 0xFFFFFFFFLL), (int)(abase >> 32), v ? (int)bbase : 0,
                         prop | (v ? (int)0x80000000 : 0));
}

// Per subdomain (once per call, one warp each): its splits sorted by hidden layer (list order
// within a layer) as packed entries, and where each layer's entries start.  Entries with a
// layer, index or sign out of range are dropped and BCROWN_ERR_ARG recorded.
__global__ void __launch_bounds__(256) k_lt_splits(int B, int L, const int* __restrict__ width, BatchView bt,
                                                   uint32_t* __restrict__ ssplit, int* __restrict__ slayer,
                                                   int* status) {
  const int b = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (b >= B) return;
  int cnt = bt.split_cnt[b];
  const int off = bt.split_off[b];
  if (cnt < 0 || cnt > BCROWN_MAX_SPLITS || off < 0) cnt = 0;   // flagged by k_lt_rowinfo
  int ly[2], pk[2];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int t = lane + 32 * h;
    ly[h] = 0;
    pk[h] = 0;
    if (t < cnt) {
      const int l = bt.split_layer[off + t];
      const int j = (int)bt.split_idx[off + t];
      const int sg = bt.split_sign[off + t];
      if (l < 1 || l > L - 1 || j < 0 || j >= width[l] || j >= (1 << 20) || (sg != 1 && sg != -1)) {
        atomicCAS(status, 0, BCROWN_ERR_ARG);
      } else {
        ly[h] = l;
        pk[h] = (int)((uint32_t)j | ((uint32_t)t << 20) | ((sg == 1 ? 1u : 0u) << 26));
      }
    }
  }
  int start = 0;
  for (int l = 0; l <= L; ++l) {
    if (lane == 0) slayer[(size_t)b * (L + 1) + l] = start;
    if (l == 0 || l == L) continue;
    const unsigned m0 = __ballot_sync(0xffffffffu, ly[0] == l), m1 = __ballot_sync(0xffffffffu, ly[1] == l);
    const unsigned below = (1u << lane) - 1u;
    if (ly[0] == l) ssplit[(size_t)b * BCROWN_MAX_SPLITS + start + __popc(m0 & below)] = (uint32_t)pk[0];
    if (ly[1] == l) ssplit[(size_t)b * BCROWN_MAX_SPLITS + start + __popc(m0) + __popc(m1 & below)] = (uint32_t)pk[1];
    start += __popc(m0) + __popc(m1);
  }
}

// lb = bbar_k + the row's partial sums, added in slot order (one warp per row: lane-strided
// sums, then a fixed shuffle tree).
__global__ void __launch_bounds__(256) k_lt_lb(Ctx cx, const float* __restrict__ bbar, float* __restrict__ lb) {
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rl = blockIdx.x * 8 + w;
  if (rl >= cx.R) return;
  const int r = cx.r0 + rl;
  const int k = r % cx.K;
  float s = 0.f;
  for (int q = lane; q < cx.S; q += 32) s += cx.cpart[(size_t)rl * cx.S + q];
  s = lt_warp_sum(s);
  if (lane == 0) {
    float v = bbar[k] + s;
    if (!isfinite(v)) {
      atomicCAS(cx.status, 0, BCROWN_ERR_NONFINITE);
      v = -INFINITY;
    }
    lb[r] = v;
  }
}

// The neurons of one hidden layer in NHWC order per property: code (0 inactive, 1 active, 2 unstable)
// | rank << 2 per neuron, the active and the unstable bits of each 8 of them, and the upper chord of
// each unstable neuron by rank.  One thread per (property, 8 channels, position); neighbouring threads
// take neighbouring positions, so the channel-major tables are read in order.
__global__ void k_lt_ntab(int P, long long H, long long hoff, int C, int HW, int Cp, long long NH, long long off,
                          Tables tb, uint32_t* __restrict__ ntab, uint16_t* __restrict__ mtab,
                          float2* __restrict__ chord) {
  const long long id = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const long long per = (long long)(Cp / 8) * HW;
  if (id >= (long long)P * per) return;
  const int p = (int)(id / per);
  const int rem = (int)(id - (long long)p * per);
  const int c8 = rem / HW, pos = rem - c8 * HW;
  uint32_t ent[8], act = 0, uns = 0;
#pragma unroll
  for (int e = 0; e < 8; ++e) {
    const int c = 8 * c8 + e;
    ent[e] = 0;
    if (c >= C) continue;
    const size_t n = (size_t)p * H + hoff + (size_t)c * HW + pos;
    const uint32_t code = tb.code[n];
    const int rk = tb.rank[n];
    ent[e] = code | ((uint32_t)max(rk, 0) << 2);
    act |= (code == CODE_ACTIVE ? 1u : 0u) << e;
    uns |= (code == CODE_UNSTABLE ? 1u : 0u) << e;
    if (code == CODE_UNSTABLE && rk >= 0) chord[(size_t)p * H + rk] = make_float2(tb.slope[n], tb.icpt[n]);
  }
  const size_t o = (size_t)p * NH + off + (size_t)pos * Cp + 8 * c8;
  *reinterpret_cast<uint4*>(ntab + o) = make_uint4(ent[0], ent[1], ent[2], ent[3]);
  *reinterpret_cast<uint4*>(ntab + o + 4) = make_uint4(ent[4], ent[5], ent[6], ent[7]);
  mtab[o / 8] = (uint16_t)(act | uns << 8);
}

constexpr int lt_smem(bool ta, int Np) {
  return 1024 + lt_stages(ta, Np) * (16384 + Np * 128) + 256 + (MAX_KP / 8) * (int)sizeof(int2) +
         MAX_NP * (int)sizeof(float) + (ta ? LtRoles<true>::EPI : LtRoles<false>::EPI) * (int)sizeof(LtList);
}
constexpr int lt_smem_max(bool ta) {
  int most = 0;
  for (int np = 16; np <= MAX_NP; np += 16) most = lt_smem(ta, np) > most ? lt_smem(ta, np) : most;
  return most;
}
static_assert(lt_smem_max(false) <= 232448 && lt_smem_max(true) <= 232448, "shared memory plan exceeds 227 KB per CTA");

}  // namespace lt

using namespace lt;

namespace {

int pad_to(int x, int m) { return (x + m - 1) / m * m; }

// NHWC map of hidden layer l (0: the input): channels, height, width, padded channels.
struct MapDims {
  int C, H, W, Cp;
  int HW() const { return H * W; }
};

MapDims map_of(const bcrown_net* net, int l) {
  MapDims m;
  if (l == 0) {
    const LayerDev& f = net->ly[0];
    m = MapDims{f.in_c, f.in_h, f.in_w, 0};
    if (f.kind != BCROWN_LAYER_CONV) m = MapDims{f.d_in, 1, 1, 0};
  } else {
    const LayerDev& f = net->ly[l - 1];
    m = f.kind == BCROWN_LAYER_CONV ? MapDims{f.out_c, f.out_h, f.out_w, 0} : MapDims{f.d_out, 1, 1, 0};
  }
  m.Cp = pad_to(m.C, 8);
  return m;
}

// Entries of a map in the NHWC neuron tables: a multiple of 64, so that 64 neurons' masks are 16-byte
// aligned, and at least 8 beyond the map.
long long nhwc_elems(const MapDims& m) { return ((long long)m.HW() * m.Cp + 8 + 63) / 64 * 64; }

// One prepared GEMM of a layer: B matrix rows [brow, brow + ntn * Np) of the layer's weight map,
// the gather table, and the pass geometry except the per-call pointers.
struct PassPrep {
  Pass p;
  int2* tab = nullptr;
};

struct LayerPrep {
  CUtensorMap mb, mf;                 // backward (phases stacked) and forward B matrices
  std::vector<PassPrep> bwd;          // one per stride phase (fc: one)
  PassPrep fwd;
};

struct LtNet {
  bool ready = false;
  std::vector<LayerPrep> ly;          // ly[i]: paper layer i (1..L-1)
  std::vector<void*> bufs;
  int S = 0;                          // partial-sum slots per row
  long long act_elems = 0;            // elements of one NHWC activation buffer per row
  int* width = nullptr;               // device [L]: d_0 .. d_{L-1}
  std::vector<float*> bnhwc;          // [l]: bias of hidden layer l in NHWC order (padded)
  std::vector<long long> nhwc_off;    // [l]: first code of hidden layer l in a property's NHWC codes
  long long NH = 0;                   // NHWC codes per property (all hidden layers, padded)
};

std::mutex g_lt_mu;
std::vector<std::pair<const bcrown_net*, LtNet*>> g_lt;

LtNet* lt_of(const bcrown_net* net) {
  std::lock_guard<std::mutex> g(g_lt_mu);
  for (auto& e : g_lt)
    if (e.first == net) return e.second;
  LtNet* t = new LtNet();
  g_lt.push_back({net, t});
  return t;
}

// Phase a of one spatial axis of a stride-s transposed convolution: taps k0 + s * d (d < nk)
// reach input rows a + s * i (i < n), whose source row is i + off - d.
struct Phase {
  int k0, nk, off, n;
};
Phase phase_of(int a, int k, int s, int pad, int in) {
  Phase c;
  c.k0 = (a + pad) % s;
  c.nk = c.k0 < k ? (k - c.k0 + s - 1) / s : 0;
  c.off = (a + pad - c.k0) / s;
  c.n = a < in ? (in - a + s - 1) / s : 0;
  return c;
}

int2 tap_entry(int elem_off, int dy, int dx) {
  return make_int2(elem_off, (int)(((uint32_t)dy & 0xffffu) | ((uint32_t)dx << 16)));
}
const int2 kNoChunk = make_int2(0, 0x8000);   // dy = -32768: no bounds test passes

int upload(LtNet* t, const void* host, size_t bytes, void** dev) {
  if (cudaMalloc(dev, bytes) != cudaSuccess) return fail(BCROWN_ERR_OOM, "layer path: device weights");
  t->bufs.push_back(*dev);
  if (cudaMemcpy(*dev, host, bytes, cudaMemcpyHostToDevice) != cudaSuccess)
    return fail(BCROWN_ERR_CUDA, "layer path: weight upload");
  return BCROWN_OK;
}

void n_tiles(int N, int* Np, int* ntn) {
  *Np = N <= MAX_NP ? pad_to(N, 16) : MAX_NP;
  *ntn = (N + *Np - 1) / *Np;
}

int prepare(bcrown_net* net, LtNet* t) {
  if (t->ready) return BCROWN_OK;
  const int L = net->L;
  t->ly.assign(L, LayerPrep());
  long long act = 0;
  for (int l = 0; l < L; ++l) {
    const MapDims m = map_of(net, l);
    act = std::max(act, (long long)m.HW() * m.Cp);
  }
  t->act_elems = pad_to((int)act, 64);
  // biases in NHWC order and the NHWC code table's layout, per hidden layer
  t->bnhwc.assign(L, nullptr);
  t->nhwc_off.assign(L, 0);
  long long nh = 0;
  for (int l = 1; l <= L - 1; ++l) {
    const MapDims m = map_of(net, l);
    const LayerDev& f = net->ly[l - 1];
    std::vector<float> bexp((size_t)f.d_out);
    if (cudaMemcpy(bexp.data(), f.b, bexp.size() * 4, cudaMemcpyDeviceToHost) != cudaSuccess)
      return fail(BCROWN_ERR_CUDA, "layer path: copy of biases");
    std::vector<float> bn((size_t)m.HW() * m.Cp + 16, 0.f);
    for (int c = 0; c < m.C; ++c)
      for (int pos = 0; pos < m.HW(); ++pos) bn[(size_t)pos * m.Cp + c] = bexp[(size_t)c * m.HW() + pos];
    void* d = nullptr;
    BC_CHECK(upload(t, bn.data(), bn.size() * 4, &d));
    t->bnhwc[l] = reinterpret_cast<float*>(d);
    t->nhwc_off[l] = nh;
    nh += nhwc_elems(m);
  }
  t->NH = nh;
  const __nv_bfloat16 zero = __float2bfloat16_rn(0.f);
  int slot = 1;   // slot 0: the top relaxation
  for (int i = L - 1; i >= 1; --i) {
    // backward slots are assigned top-down, in the order the passes run
    const LayerDev& l = net->ly[i - 1];
    const MapDims mi = map_of(net, i), mo = map_of(net, i - 1);   // GEMM source, output
    std::vector<float> w(l.kind == BCROWN_LAYER_CONV ? (size_t)l.out_c * l.in_c * l.k * l.k
                                                     : (size_t)l.d_out * l.d_in);
    if (cudaMemcpy(w.data(), l.W, w.size() * 4, cudaMemcpyDeviceToHost) != cudaSuccess)
      return fail(BCROWN_ERR_CUDA, "layer path: copy of weights");
    LayerPrep& P = t->ly[i];
    auto finish_pass = [&](PassPrep& pp, std::vector<int2>& tab) -> int {
      void* d = nullptr;
      BC_CHECK(upload(t, tab.data(), tab.size() * sizeof(int2), &d));
      pp.tab = reinterpret_cast<int2*>(d);
      pp.p.tab = pp.tab;
      // The A operand by TMA where an M tile is one box of the NHWC source (whole rows of the
      // pass's position grid, or whole grids of consecutive subdomain rows) and each K block is
      // one tap's 64-channel block (source channels a multiple of 64).  A position step ms > 1
      // (a strided convolution's forward pass) is the box's traversal step in x and y: the box
      // spans ms times the positions it holds.
      Pass& q = pp.p;
      int bw = 0, bh = 0, br = 0;
      const bool narrow = q.Cps == 8 && q.nkb <= 16;   // 8 channels: one box per tap
      if (q.ms >= 1 && q.ms <= 8 && (q.Cps % 64 == 0 || narrow) && q.nJ > 0 && q.Pm > 0) {
        if (q.Pm % 128 == 0) {
          if (q.nJ <= 128 && 128 % q.nJ == 0) bw = q.nJ, bh = 128 / q.nJ, br = 1;
          else if (q.nJ % 128 == 0) bw = 128, bh = 1, br = 1;
        } else if (128 % q.Pm == 0 && q.Pm % q.nJ == 0) {
          bw = q.nJ, bh = q.Pm / q.nJ, br = 128 / q.Pm;
        }
      }
      if (bw > 0 && bw * bh * br == 128 && bw * q.ms <= 256 && bh * q.ms <= 256 && (size_t)q.nkb * 8 == tab.size() &&
          narrow) {
        std::vector<int4> kt(tab.size());
        for (size_t kc = 0; kc < tab.size(); ++kc) {
          const int dy = (int)(short)(tab[kc].y & 0xffff), dx = tab[kc].y >> 16;
          const bool used = dy != -32768;
          kt[kc] = make_int4(0, used ? dy : 0, used ? dx : 0, used ? 1 : 0);
        }
        void* dk = nullptr;
        BC_CHECK(upload(t, kt.data(), kt.size() * sizeof(int4), &dk));
        q.ktab = reinterpret_cast<const int4*>(dk);
        q.ta = 8, q.bw = bw, q.bh = bh, q.br = br;
      } else if (bw > 0 && bw * bh * br == 128 && bw * q.ms <= 256 && bh * q.ms <= 256 &&
                 (size_t)q.nkb * 8 == tab.size()) {
        const int cpb = q.Cps / 64;
        std::vector<int4> kt((size_t)q.nkb);
        for (int kb = 0; kb < q.nkb; ++kb) {
          const int2 e = tab[(size_t)kb * 8];
          const int dy = (int)(short)(e.y & 0xffff), dx = e.y >> 16;
          const bool used = dy != -32768;
          kt[kb] = make_int4((kb % cpb) * 64, used ? dy : 0, used ? dx : 0, used ? 1 : 0);
        }
        void* dk = nullptr;
        BC_CHECK(upload(t, kt.data(), kt.size() * sizeof(int4), &dk));
        q.ktab = reinterpret_cast<const int4*>(dk);
        q.ta = 4, q.bw = bw, q.bh = bh, q.br = br;
      }
      return BCROWN_OK;
    };
    if (l.kind == BCROWN_LAYER_CONV) {
      const int s = l.stride, k = l.k;
      const int T = (k + s - 1) / s;
      // backward: per phase (a, b), N = input channels, K = (dy, dx, output channel)
      int Np = 0, ntn = 0;
      n_tiles(mo.C, &Np, &ntn);
      const int kp = pad_to(T * T * mi.Cp, 64);
      std::vector<__nv_bfloat16> wb((size_t)s * s * Np * kp, zero);
      for (int a = 0; a < s; ++a)
        for (int bb = 0; bb < s; ++bb) {
          const Phase py = phase_of(a, k, s, l.pad, l.in_h), px = phase_of(bb, k, s, l.pad, l.in_w);
          const int ph = a * s + bb;
          PassPrep pp;
          Pass& q = pp.p;
          q.Pm = py.n * px.n;
          q.nJ = px.n;
          q.N = mo.C;
          q.Np = Np;
          q.ntn = ntn;
          // the phase's own taps (a stride-2 3x3 layer's phases have 1, 2, 2 and 4)
          const int kph = std::max(64, pad_to(py.nk * px.nk * mi.Cp, 64));
          q.nkb = kph / 64;
          q.brow = ph * Np;
          q.Hs = mi.H;
          q.Ws = mi.W;
          q.Cps = mi.Cp;
          q.ms = 1;
          q.cy = py.off;
          q.cx = px.off;
          q.kchunks = kph / 8;
          q.oa = a;
          q.ob = bb;
          q.os = s;
          q.Wo = mo.W;
          q.npos = 0;
          q.Co = mo.C;
          q.HWo = mo.HW();
          q.Cpo = mo.Cp;
          q.layer = i - 1;
          q.bnhwc = i >= 2 ? t->bnhwc[i - 1] : nullptr;
          std::vector<int2> tab((size_t)kph / 8, kNoChunk);
          for (int dy = 0; dy < py.nk; ++dy)
            for (int dx = 0; dx < px.nk; ++dx) {
              const int tap = dy * px.nk + dx;
              for (int c8 = 0; c8 < mi.Cp / 8; ++c8)
                tab[(size_t)tap * (mi.Cp / 8) + c8] = tap_entry((-dy * mi.W - dx) * mi.Cp + 8 * c8, -dy, -dx);
              const int ky = py.k0 + s * dy, kx = px.k0 + s * dx;
              for (int co = 0; co < l.out_c; ++co)
                for (int ci = 0; ci < l.in_c; ++ci)
                  wb[((size_t)ph * Np + ci) * kp + (size_t)tap * mi.Cp + co] =
                      __float2bfloat16_rn(w[(((size_t)co * l.in_c + ci) * k + ky) * k + kx]);
            }
          if (q.Pm > 0) {
            BC_CHECK(finish_pass(pp, tab));
            q.slot0 = slot;
            slot += (q.Pm % 32 == 0) ? ntn * q.Pm / 32 : ntn * q.Pm;
            P.bwd.push_back(pp);
          }
        }
      void* db = nullptr;
      BC_CHECK(upload(t, wb.data(), wb.size() * 2, &db));
      BC_CHECK(encode_map(&P.mb, db, s * s * Np, kp, Np));
      // forward: N = output channels, K = (ky, kx, input channel)
      int Npf = 0, ntnf = 0;
      n_tiles(mi.C, &Npf, &ntnf);
      const int kpf = pad_to(k * k * mo.Cp, 64);
      std::vector<__nv_bfloat16> wf((size_t)ntnf * Npf * kpf, zero);
      std::vector<int2> tab((size_t)kpf / 8, kNoChunk);
      for (int ky = 0; ky < k; ++ky)
        for (int kx = 0; kx < k; ++kx) {
          const int tap = ky * k + kx;
          for (int c8 = 0; c8 < mo.Cp / 8; ++c8)
            tab[(size_t)tap * (mo.Cp / 8) + c8] = tap_entry((ky * mo.W + kx) * mo.Cp + 8 * c8, ky, kx);
          for (int co = 0; co < l.out_c; ++co)
            for (int ci = 0; ci < l.in_c; ++ci)
              wf[(size_t)co * kpf + (size_t)tap * mo.Cp + ci] =
                  __float2bfloat16_rn(w[(((size_t)co * l.in_c + ci) * k + ky) * k + kx]);
        }
      Pass& q = P.fwd.p;
      q.Pm = mi.HW();
      q.nJ = mi.W;
      q.N = mi.C;
      q.Np = Npf;
      q.ntn = ntnf;
      q.nkb = kpf / 64;
      q.brow = 0;
      q.Hs = mo.H;
      q.Ws = mo.W;
      q.Cps = mo.Cp;
      q.ms = s;
      q.cy = -l.pad;
      q.cx = -l.pad;
      q.kchunks = kpf / 8;
      q.oa = 0;
      q.ob = 0;
      q.os = 1;
      q.Wo = mi.W;
      q.npos = 0;
      q.Co = mi.C;
      q.HWo = mi.HW();
      q.Cpo = mi.Cp;
      q.layer = i;
      q.bnhwc = t->bnhwc[i];
      q.slot0 = 0;
      BC_CHECK(finish_pass(P.fwd, tab));
      void* df = nullptr;
      BC_CHECK(upload(t, wf.data(), wf.size() * 2, &df));
      BC_CHECK(encode_map(&P.mf, df, ntnf * Npf, kpf, Npf));
    } else {
      // fully connected: input = map mo (NHWC index p * Cp + c of neuron c * HW + p), output a vector
      const int din_n = mo.HW() * mo.Cp;   // NHWC-padded input length
      // backward: N = din_n (npos), K = output neurons (padded to 8, then 64)
      int Np = 0, ntn = 0;
      n_tiles(din_n, &Np, &ntn);
      const int kp = pad_to(mi.Cp, 64);
      std::vector<__nv_bfloat16> wb((size_t)ntn * Np * kp, zero);
      for (int o = 0; o < l.d_out; ++o)
        for (int c = 0; c < mo.C; ++c)
          for (int p = 0; p < mo.HW(); ++p)
            wb[((size_t)p * mo.Cp + c) * kp + o] = __float2bfloat16_rn(w[(size_t)o * l.d_in + (size_t)c * mo.HW() + p]);
      PassPrep pp;
      Pass& q = pp.p;
      q.Pm = 1;
      q.nJ = 1;
      q.N = din_n;
      q.Np = Np;
      q.ntn = ntn;
      q.nkb = kp / 64;
      q.brow = 0;
      q.Hs = 1;
      q.Ws = 1;
      q.Cps = mi.Cp;
      q.ms = 1;
      q.cy = 0;
      q.cx = 0;
      q.oa = 0;
      q.ob = 0;
      q.os = 1;
      q.Wo = 1;
      q.npos = 1;
      q.Co = mo.C;
      q.HWo = mo.HW();
      q.Cpo = mo.Cp;
      q.layer = i - 1;
      q.bnhwc = i >= 2 ? t->bnhwc[i - 1] : nullptr;
      q.kchunks = mi.Cp / 8;   // K chunks past the layer's padded width read as zero
      q.tab = nullptr;
      q.ta = 2;   // the linear source: the A operand by TMA, 64 x 128-row boxes
      q.slot0 = slot;
      slot += ntn;
      P.bwd.push_back(pp);
      void* db = nullptr;
      BC_CHECK(upload(t, wb.data(), wb.size() * 2, &db));
      BC_CHECK(encode_map(&P.mb, db, ntn * Np, kp, Np));
      // forward: N = output neurons, K = din_n (padded to 64)
      int Npf = 0, ntnf = 0;
      n_tiles(mi.C, &Npf, &ntnf);
      const int kpf = pad_to(din_n, 64);
      std::vector<__nv_bfloat16> wf((size_t)ntnf * Npf * kpf, zero);
      for (int o = 0; o < l.d_out; ++o)
        for (int c = 0; c < mo.C; ++c)
          for (int p = 0; p < mo.HW(); ++p)
            wf[(size_t)o * kpf + (size_t)p * mo.Cp + c] = __float2bfloat16_rn(w[(size_t)o * l.d_in + (size_t)c * mo.HW() + p]);
      Pass& f = P.fwd.p;
      f = q;
      f.N = mi.C;
      f.Np = Npf;
      f.ntn = ntnf;
      f.nkb = kpf / 64;
      f.Cps = mo.Cp;
      f.kchunks = din_n / 8;
      f.tab = nullptr;
      f.ta = 2;
      f.npos = 0;
      f.Co = mi.C;
      f.HWo = 1;
      f.Cpo = mi.Cp;
      f.Wo = 1;
      f.layer = i;
      f.bnhwc = t->bnhwc[i];
      f.slot0 = 0;
      void* df = nullptr;
      BC_CHECK(upload(t, wf.data(), wf.size() * 2, &df));
      BC_CHECK(encode_map(&P.mf, df, ntnf * Npf, kpf, Npf));
    }
  }
  t->S = slot;
  {
    std::vector<int> wd(net->d.begin(), net->d.begin() + L);
    void* d = nullptr;
    BC_CHECK(upload(t, wd.data(), wd.size() * sizeof(int), &d));
    t->width = reinterpret_cast<int*>(d);
  }
  const int smem_g = lt_smem_max(false), smem_t = lt_smem_max(true);
  BC_CUDA(cudaFuncSetAttribute(k_lt<EPI_RELAX, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_g));
  BC_CUDA(cudaFuncSetAttribute(k_lt<EPI_CONCRETIZE, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_g));
  BC_CUDA(cudaFuncSetAttribute(k_lt<EPI_FWD, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_g));
  BC_CUDA(cudaFuncSetAttribute(k_lt<EPI_RELAX, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_t));
  BC_CUDA(cudaFuncSetAttribute(k_lt<EPI_CONCRETIZE, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_t));
  BC_CUDA(cudaFuncSetAttribute(k_lt<EPI_FWD, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_t));
  t->ready = true;
  return BCROWN_OK;
}

int launch_pass(bcrown_net* net, const CUtensorMap& mB, Pass q, int mode, const Ctx& cx, cudaStream_t s) {
  q.M = (long long)cx.R * q.Pm;
  if (q.M <= 0) return BCROWN_OK;
  int dev = 0, sms = 148;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  q.dPm.set(q.Pm);
  q.dnJ.set(q.nJ);
  q.dntn.set(q.ntn);
  q.dHWo.set(q.HWo);
  const long long ntiles = (q.M + 127) / 128 * q.ntn;
  const int grid = (int)std::min<long long>(ntiles, sms);
  const int smem = lt_smem(q.ta != 0, q.Np);
  ProfScope pr(net, BCROWN_PROF_LAYER_GEMM, s);
  // the A operand's map for this launch (the source buffer and the rows of this chunk)
  CUtensorMap mA = mB;   // unused by the gathering kernel
  if (q.ta == 4 || q.ta == 8) {
    const cuuint64_t dims[4] = {(cuuint64_t)q.Cps, (cuuint64_t)q.Ws, (cuuint64_t)q.Hs, (cuuint64_t)cx.R};
    const cuuint64_t strides[3] = {(cuuint64_t)q.Cps * 2, (cuuint64_t)q.Ws * q.Cps * 2, (cuuint64_t)q.src_stride * 2};
    // a strided pass: boxes of ms bw x ms bh source positions, every ms-th one loaded (bw x bh)
    const cuuint32_t box[4] = {q.ta == 8 ? 8u : 64u, (cuuint32_t)(q.bw * q.ms), (cuuint32_t)(q.bh * q.ms),
                               (cuuint32_t)q.br};
    const cuuint32_t es[4] = {1, (cuuint32_t)q.ms, (cuuint32_t)q.ms, 1};
    BC_CHECK(encode_map_nd(&mA, const_cast<__nv_bfloat16*>(q.src), 4, dims, strides, box, es, q.ta == 4));
  } else if (q.ta == 2) {
    const cuuint64_t dims[2] = {(cuuint64_t)q.kchunks * 8, (cuuint64_t)cx.R};
    const cuuint64_t strides[1] = {(cuuint64_t)q.src_stride * 2};
    const cuuint32_t box[2] = {64, 128};
    BC_CHECK(encode_map_nd(&mA, const_cast<__nv_bfloat16*>(q.src), 2, dims, strides, box));
  }
  if (q.ta) {
    if (mode == EPI_RELAX) k_lt<EPI_RELAX, true><<<grid, LtRoles<true>::THREADS, smem, s>>>(mB, mA, q, cx);
    else if (mode == EPI_CONCRETIZE) k_lt<EPI_CONCRETIZE, true><<<grid, LtRoles<true>::THREADS, smem, s>>>(mB, mA, q, cx);
    else k_lt<EPI_FWD, true><<<grid, LtRoles<true>::THREADS, smem, s>>>(mB, mA, q, cx);
  } else {
    if (mode == EPI_RELAX) k_lt<EPI_RELAX, false><<<grid, LtRoles<false>::THREADS, smem, s>>>(mB, mA, q, cx);
    else if (mode == EPI_CONCRETIZE) k_lt<EPI_CONCRETIZE, false><<<grid, LtRoles<false>::THREADS, smem, s>>>(mB, mA, q, cx);
    else k_lt<EPI_FWD, false><<<grid, LtRoles<false>::THREADS, smem, s>>>(mB, mA, q, cx);
  }
  ++g_launches;
  BC_CUDA(cudaGetLastError());
  return BCROWN_OK;
}

}  // namespace

// Per-row sizes of the workspace: the NHWC activation buffer (elements) and an upper bound of the
// partial-sum slots (one per position block and column group of every backward pass), and the
// rows per chunk for a 16 GB target.
static void plan_sizes(const bcrown_net* net, int R, long long* act, long long* S, long long* Rc) {
  long long a = 0, sl = 1;
  for (int l = 0; l < net->L; ++l) {
    const MapDims m = map_of(net, l);
    a = std::max(a, (long long)m.HW() * m.Cp);
  }
  for (int i = 1; i <= net->L - 1; ++i) {
    const MapDims mo = map_of(net, i - 1);
    sl += 2LL * mo.HW() * std::max(1, (mo.Cp + MAX_NP - 1) / MAX_NP) + 2LL * (((long long)mo.HW() * mo.Cp + MAX_NP - 1) / MAX_NP);
  }
  *act = (a + 63) / 64 * 64;
  *S = sl;
  const size_t per_row = (size_t)2 * *act * 2 + (size_t)sl * 4;
  const size_t target = size_t(16) << 30;
  *Rc = std::max<long long>(1, std::min<long long>(std::max(R, 1), (long long)(target / per_row)));
}

bool lt_supported(const bcrown_net* net) {
  if (net->L < 2) return false;
  for (int i = 1; i <= net->L - 1; ++i) {
    const LayerDev& l = net->ly[i - 1];
    const MapDims mi = map_of(net, i), mo = map_of(net, i - 1);
    if (l.kind == BCROWN_LAYER_CONV) {
      if (l.in_c > MAX_NP || l.out_c > MAX_NP) return false;
      const int T = (l.k + l.stride - 1) / l.stride;
      if (pad_to(T * T * mi.Cp, 64) > MAX_KP || pad_to(l.k * l.k * mo.Cp, 64) > MAX_KP) return false;
    } else {
      if (pad_to(mi.Cp, 64) > MAX_KP) return false;   // backward K
      if ((long long)mo.HW() * mo.Cp > 65536 || l.d_out > 65536) return false;
    }
    if ((long long)mi.HW() * mi.Cp > (1LL << 24)) return false;
  }
  int dev = 0, major = 0, minor = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return false;
  cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev);
  cudaDeviceGetAttribute(&minor, cudaDevAttrComputeCapabilityMinor, dev);
  cudaGetLastError();
  return major == 10 && minor == 3;
}

size_t lt_workspace_bytes(const bcrown_net* net, int R, int P, int64_t n_alpha, bool grad) {
  long long act, S, Rc;
  plan_sizes(net, R, &act, &S, &Rc);
  long long nh = 0;
  for (int l = 1; l <= net->L - 1; ++l) {
    const MapDims m = map_of(net, l);
    nh += nhwc_elems(m);
  }
  const size_t B = (size_t)R / std::max(net->K, 1);
  size_t bytes = align_up((size_t)Rc * act * 2) * 2 + align_up((size_t)Rc * S * 4);
  bytes += align_up((size_t)R * 16) + align_up(B * BCROWN_MAX_SPLITS * 4) + align_up(B * (net->L + 1) * 4);
  bytes += align_up((size_t)std::max(P, 1) * nh * 4) + align_up((size_t)std::max(P, 1) * nh / 4) +
           align_up((size_t)std::max(P, 1) * std::max(net->H, 1) * 8);
  if (grad) bytes += align_up((size_t)std::max<int64_t>(n_alpha, 1) * 2);
  return bytes;
}

int lt_bound(bcrown_net* net, const bcrown_domain* dom, const bcrown_batch* bt, const Tables& tb, char* ws,
             size_t ws_bytes, bool grad, const float* alpha, const float* beta, float* lb, float* dalpha,
             float* dbeta, cudaStream_t s) {
  LtNet* t = lt_of(net);
  BC_CHECK(prepare(net, t));
  const int K = net->K, L = net->L;
  const int R = bt->B * K;
  if (R == 0) return BCROWN_OK;
  if (ws_bytes < lt_workspace_bytes(net, R, dom->n_props, bt->n_alpha, grad))
    return fail(BCROWN_ERR_OOM, "layer path: workspace");
  long long act_b, S_b, Rc;
  plan_sizes(net, R, &act_b, &S_b, &Rc);
  if (act_b != t->act_elems || S_b < t->S) return fail(BCROWN_ERR_ARG, "layer path: inconsistent plan");
  Arena ar{ws};
  __nv_bfloat16* act[2];
  act[0] = ar.take<__nv_bfloat16>((size_t)Rc * t->act_elems);
  act[1] = ar.take<__nv_bfloat16>((size_t)Rc * t->act_elems);
  float* cpart = ar.take<float>((size_t)Rc * S_b);
  int4* rowinfo = ar.take<int4>((size_t)R);
  uint32_t* ssplit = ar.take<uint32_t>((size_t)bt->B * BCROWN_MAX_SPLITS);
  int* slayer = ar.take<int>((size_t)bt->B * (L + 1));
  uint32_t* ntab = ar.take<uint32_t>((size_t)dom->n_props * t->NH);
  uint16_t* mtab = ar.take<uint16_t>((size_t)dom->n_props * t->NH / 8);
  float2* chord = ar.take<float2>((size_t)dom->n_props * std::max(net->H, 1));
  __nv_bfloat16* stash = grad ? ar.take<__nv_bfloat16>((size_t)std::max<int64_t>(bt->n_alpha, 1)) : nullptr;
  if (ar.off > ws_bytes) return fail(BCROWN_ERR_OOM, "layer path: workspace plan");
  Ctx cx;
  cx.K = K;
  cx.dK.set(K);
  cx.P = dom->n_props;
  cx.H = net->H;
  cx.d0 = net->d[0];
  cx.S = t->S;
  cx.bt = BatchView{bt->B, bt->prop_of, bt->split_off, bt->split_cnt, bt->split_layer, bt->split_idx, bt->split_sign,
                    bt->alpha_off};
  cx.tb = tb;
  cx.x_lo = dom->x_lo;
  cx.x_hi = dom->x_hi;
  cx.alpha = alpha;
  cx.beta = beta;
  cx.n_alpha = bt->n_alpha;
  cx.n_beta = bt->n_beta;
  cx.dalpha = dalpha;
  cx.dbeta = dbeta;
  cx.stash = stash;
  cx.cpart = cpart;
  cx.status = net->status;
  cx.rowinfo = rowinfo;
  cx.ssplit = ssplit;
  cx.slayer = slayer;
  cx.L = L;
  cx.NH = t->NH;
  cx.chord = chord;
  // the properties' neurons in NHWC order and their chords by rank, once per call
  for (int l = 1; l <= L - 1; ++l) {
    const MapDims m = map_of(net, l);
    const long long n = (long long)dom->n_props * (m.Cp / 8) * m.HW();
    k_lt_ntab<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(dom->n_props, net->H, net->hoff[l - 1], m.C, m.HW(), m.Cp,
                                                         t->NH, t->nhwc_off[l], tb, ntab, mtab, chord);
    ++g_launches;
  }
  // the rows' alpha / beta offsets and the subdomains' splits sorted by layer, once per call
  k_lt_rowinfo<<<(R + 255) / 256, 256, 0, s>>>(R, K, dom->n_props, cx.bt, tb.U, bt->n_alpha, rowinfo, net->status);
  k_lt_splits<<<(bt->B * 32 + 255) / 256, 256, 0, s>>>(bt->B, L, t->width, cx.bt, ssplit, slayer, net->status);
  g_launches += 2;
  const long long stride = t->act_elems;
  for (long long r0 = 0; r0 < R; r0 += Rc) {
    cx.r0 = (int)r0;
    cx.R = (int)std::min<long long>(Rc, R - r0);
    // top: Lambda^(L-1) into act[0]
    {
      ProfScope pr(net, BCROWN_PROF_RELAX, s);
      const MapDims mt = map_of(net, L - 1);
      k_lt_top<<<(cx.R + 7) / 8, 256, 0, s>>>(cx, L - 1, net->hoff[L - 2], mt.C, mt.HW(), mt.Cp, net->Wbar,
                                              net->ly[L - 2].b, act[0], stride);
      ++g_launches;
    }
    int cur = 0;
    for (int i = L - 1; i >= 1; --i) {
      const LayerPrep& P = t->ly[i];
      for (const PassPrep& pp : P.bwd) {
        Pass q = pp.p;
        q.ntab = i >= 2 ? ntab + t->nhwc_off[i - 1] : nullptr;
        q.mtab = i >= 2 ? mtab + t->nhwc_off[i - 1] / 8 : nullptr;
        q.src = act[cur];
        q.src_stride = stride;
        q.dst = act[cur ^ 1];
        q.dst_stride = stride;
        BC_CHECK(launch_pass(net, P.mb, q, i == 1 ? EPI_CONCRETIZE : EPI_RELAX, cx, s));
      }
      cur ^= 1;
    }
    {
      ProfScope pr(net, BCROWN_PROF_CONCRETIZE, s);
      k_lt_lb<<<(cx.R + 7) / 8, 256, 0, s>>>(cx, net->bbar, lb);
      ++g_launches;
    }
    if (!grad) continue;
    // adjoint: x* is in act[cur]
    for (int i = 1; i <= L - 1; ++i) {
      const LayerPrep& P = t->ly[i];
      Pass q = P.fwd.p;
      q.ntab = ntab + t->nhwc_off[i];
      q.mtab = mtab + t->nhwc_off[i] / 8;
      q.src = act[cur];
      q.src_stride = stride;
      q.dst = i < L - 1 ? act[cur ^ 1] : nullptr;
      q.dst_stride = stride;
      BC_CHECK(launch_pass(net, P.mf, q, EPI_FWD, cx, s));
      cur ^= 1;
    }
  }
  BC_CUDA(cudaGetLastError());
  return BCROWN_OK;
}

void lt_release(const bcrown_net* net) {
  std::lock_guard<std::mutex> g(g_lt_mu);
  for (size_t i = 0; i < g_lt.size(); ++i)
    if (g_lt[i].first == net) {
      for (void* b : g_lt[i].second->bufs) cudaFree(b);
      delete g_lt[i].second;
      g_lt.erase(g_lt.begin() + i);
      return;
    }
}

}  // namespace bcrown
