// Fused tensor-core bound pass for fully connected ReLU networks (sm_103a: tcgen05 + TMA).
//
// One persistent CTA per SM walks tiles of TR = 16, 32 or 64 rows (row = subdomain x spec).  For a
// tile, the whole backward recursion of Theorem 3.1 (Eq. definition_A) runs on chip:
//
//   A^(i-1)^T = W^(i)^T Lambda^(i)^T      (tcgen05.mma, M = 128 output neurons, N = TR rows,
//                                          K = 16; BF16 operands, FP32 accumulator in TMEM)
//
// The weight tile is the MMA's A operand (loaded by TMA, 128B swizzle, K-major) and the
// activations Lambda^T are its B operand (written to shared memory by the epilogue in the
// same swizzled layout).  Putting neurons on TMEM lanes makes every epilogue access to
// alpha, the per-neuron tables, the gradients and the stash coalesced across a warp.
//
// The epilogue (16 warps) reads the accumulator with tcgen05.ld, applies the relaxation of
// Lemma 2.1 / Eq. definition_D (split overriding stability), the beta shift and the bias
// sums (Lambda = A D + beta S; c += Lambda b + A lambda), and writes Lambda^(i-1) in BF16
// as the next contraction's operand.  The last contraction is concretised over the box
// (Eq. beta_crown_lp).  With a gradient requested the adjoint pass follows in the same
// launch: zhat^(i) = W^(i) h^(i-1) + b^(i) along h^(0) = x*, dalpha = A zhat, dbeta = S zhat,
// h = D zhat + lambda.  The kernel writes the gradients only: the projected Adam step
// (Appendix C.1) and the per-row best tracking run afterwards in a separate element-wise
// kernel over alpha and beta.
//
// Roles: warps 0-15 epilogue, warp 16 TMA producer, warp 17 MMA issuer.
// Every mbarrier wait is bounded; on expiry the kernel records BCROWN_ERR_TIMEOUT, stops
// issuing work, waits (bounded) for its copies in flight, frees TMEM and returns.
#include <cuda.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <atomic>
#include <cstring>

#include "fused_tc.cuh"
#include "tc_ptx.cuh"

namespace bcrown {

extern std::atomic<long long> g_launches;

namespace tc {

constexpr int MCH = 128;          // neurons per M chunk = MMA M
constexpr int NSLOT = 4;          // activation (B operand) slots of one K pair (2 blocks of 64): an
                                  // operand of up to 256 neurons takes the half (slots 2h, 2h + 1)
                                  // the one before it does not; x* streams through its half
constexpr int NSTAGE = 3;         // weight (A operand) ring, of K pairs
constexpr int NACC = 4;           // accumulator ring (TR columns each)
constexpr int NFACC = 2;          // the forward contraction of layer 1 (all its M chunks at once)
constexpr int XLAG = 3;           // x* pair e is contracted after chunk e + XLAG of the concretisation
constexpr int STAGE_BYTES = MCH * 128;   // 16 KB: one K block of a stage
constexpr int NEPI = 16;                 // epilogue warps
constexpr int TMA_WARP = 16, MMA_WARP = 17;
constexpr int NTHREADS = 18 * 32;
constexpr int MAXL = 9;
constexpr int MAX_D0 = 1024;
constexpr int MAX_MASK_WORDS = 48;       // sum over hidden layers of ceil(d_i/32)
static_assert(MAX_MASK_WORDS % 8 == 0, "set-up step 3 splits the mask words over 8 threads per row");
constexpr int MAX_H = MAX_MASK_WORDS * 32;  // hidden neurons whose tables a tile stages
constexpr int MAX_HIDDEN = 256;

// TR: rows per tile (subdomain x spec) = MMA N.  A K block of an operand is TR rows of 128 bytes.
template <int TR>
struct Smem {
  uint8_t act[NSLOT][2 * TR * 128];      // TR = 64: 64 KB, 1024-aligned blocks
  uint8_t w[NSTAGE][2 * STAGE_BYTES];    // 96 KB
  uint32_t smask[MAX_MASK_WORDS][TR];    // split present, [word][row]: a warp reads its 16 rows at once
  unsigned long long wrows[MAX_MASK_WORDS];  // rows with any split in mask word w
  float part[4][TR];                     // lb partial sums per lane quadrant
  alignas(16) long long abase[TR];       // first alpha of the row
  long long bbase[TR];                   // first beta of the row
  int rowid[TR];                         // global row of each tile slot (-1: empty)
  int spec[TR];
  int valid[TR];
  int scnt[TR];                          // the row's split count and first split entry
  int soff[TR];
  uint8_t sorig[TR][BCROWN_MAX_SPLITS];  // the row's splits in (mask word, bit) order: list position
  float sbeta[TR][BCROWN_MAX_SPLITS];    //   and beta S (beta clamped at 0; the sign bit tells S)
  uint8_t wfirst[MAX_MASK_WORDS][TR];    // splits of the row in mask words before w
  uint32_t tcode[MAX_H];                 // the tile's property: code << 16 | unstable rank, per hidden neuron
  float tslope[MAX_H];                   //   upper chord slope
  float ticpt[MAX_H];                    //   upper chord intercept
  unsigned long long vrows;              // tile slots holding a valid row
  uint64_t act_full[NSLOT], act_empty[NSLOT];
  uint64_t w_full[NSTAGE], w_empty[NSTAGE];
  uint64_t acc_full[NACC], acc_empty[NACC];
  uint64_t facc_full;                    // the forward contraction of layer 1
  uint64_t epi;   // epilogue-wide barrier (NEPI warp arrivals per phase)
  uint64_t done;
  uint32_t tmem_base;
  int abort_flag;
};

static_assert(sizeof(Smem<64>) + 1024 <= 232448, "shared memory plan exceeds 227 KB per CTA");

struct Args {
  int L, K, P, H, R;
  int tiles;                          // with one property: its tiles, rows in order (no plan)
  const int* n_tiles;                 // tiles to process (written by the row planner; null: one property)
  const int* tile_prop;               // [tile] property of every row of the tile
  const int* rowmap;                  // [tile][TR] global row of each slot, -1 when empty
  int d[MAXL + 1];
  long long hoff[MAXL + 1];           // first global hidden index of layer i (1-based)
  int woff[MAXL + 1];                 // first mask word of layer i
  int mask_words;
  const float* bias[MAXL + 1];
  const float* Wbar;
  const float* bbar;
  BatchView bt;
  Tables tb;
  const float* x_lo;
  const float* x_hi;
  const float* alpha;
  const float* beta;
  int64_t n_alpha, n_beta;
  float* lb;
  float* dalpha;
  __nv_bfloat16* dalpha16;            // MODE 2: dlb/dalpha rounded to BF16 (optimiser input)
  float* dbeta;
  __nv_bfloat16* stash;               // [tile][H][TR]: A^(i) of the backward pass, per neuron
  int* status;
  int box_bwd[MAXL + 1];
  int box_fwd[MAXL + 1];
};

struct Maps {
  CUtensorMap bwd[MAXL + 1];   // Wt^(i): [d_{i-1}][Kp(d_i)] bf16, rows = output neurons of the backward
  CUtensorMap fwd[MAXL + 1];   // W^(i):  [d_i][Kp(d_{i-1})] bf16, rows = output neurons of the forward
};

// ------------------------------------------------------------------------------------------
// PTX helpers
// ------------------------------------------------------------------------------------------

// Bounded wait (about 2 s of SM clock); on expiry records a timeout and raises the abort flag.
// Inlined: as a called function it cost the single-thread MMA and TMA loops ~0.2 us per wait.
template <class SM>
__device__ __forceinline__ bool mbar_wait(uint64_t* b, uint32_t parity, SM* sm, int* status) {
  if (mbar_try(b, parity)) return true;
  long long t0 = clock64();
  while (true) {
    if (mbar_try_sleep(b, parity, 20000u)) return true;
    if (*(volatile int*)&sm->abort_flag) return false;
    if (clock64() - t0 > 4000000000LL) {
      atomicCAS(status, 0, BCROWN_ERR_TIMEOUT);
      *(volatile int*)&sm->abort_flag = 1;
      return false;
    }
  }
}
// The TMA and the MMA warp (one warp each) wait with all lanes.
template <class SM>
__device__ __forceinline__ bool mbar_wait_all(uint64_t* b, uint32_t parity, SM* sm, int* status) {
  return mbar_wait_together(b, parity, [&] { return *(volatile int*)&sm->abort_flag != 0; },
                            [&] {
                              atomicCAS(status, 0, BCROWN_ERR_TIMEOUT);
                              *(volatile int*)&sm->abort_flag = 1;
                            });
}
// Wait by a whole warp: one lane polls the barrier (512 polling threads would flood the
// shared-memory pipe every other warp needs), then the warp reconverges.
template <class SM>
__device__ __forceinline__ bool mbar_wait_warp(uint64_t* b, uint32_t parity, SM* sm, int* status) {
  __syncwarp();
  int ok = 1;
  if ((threadIdx.x & 31) == 0) ok = mbar_wait(b, parity, sm, status) ? 1 : 0;
  ok = __shfl_sync(0xffffffffu, ok, 0);
  __syncwarp();
  return ok != 0;
}
// Barrier among the 16 epilogue warps built on an mbarrier, so that a warp that gives up
// after a timeout cannot leave the others blocked: every wait here is bounded.
template <class SM>
__device__ __forceinline__ bool epi_sync(SM* sm, uint32_t& seq, int* status) {
  __syncwarp();
  if ((threadIdx.x & 31) == 0) mbar_arrive(&sm->epi);
  const bool ok = mbar_wait_warp(&sm->epi, seq & 1, sm, status);
  ++seq;
  return ok;
}

// Loads issued where they are written (volatile asm keeps them ahead of the barrier waits that
// follow, instead of letting the compiler sink them to their first use); 0 when pred is false.
__device__ __forceinline__ float ldg_f32(const float* p, bool pred) {
  float v;
  asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %2, 0;\n\tmov.f32 %0, 0f00000000;\n\t@q ld.global.f32 %0, [%1];\n\t}"
               : "=f"(v)
               : "l"(p), "r"((uint32_t)pred)
               : "memory");
  return v;
}
// Four of them under one predicate.
__device__ __forceinline__ void ldg4_f32(const float* p0, const float* p1, const float* p2, const float* p3, bool pred,
                                         float* v) {
  asm volatile(
      "{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %8, 0;\n\tmov.f32 %0, 0f00000000;\n\tmov.f32 %1, 0f00000000;\n\t"
      "mov.f32 %2, 0f00000000;\n\tmov.f32 %3, 0f00000000;\n\t@q ld.global.f32 %0, [%4];\n\t@q ld.global.f32 %1, [%5];\n\t"
      "@q ld.global.f32 %2, [%6];\n\t@q ld.global.f32 %3, [%7];\n\t}"
      : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3])
      : "l"(p0), "l"(p1), "l"(p2), "l"(p3), "r"((uint32_t)pred)
      : "memory");
}

// Sum of v[r] over the 32 lanes of a warp, r = 0 .. N - 1 (N = 4, 8 or 16), scattered: lanes
// (32 / N) r .. (32 / N) (r + 1) - 1 hold the sum for r.  The lanes are added in the order of the
// butterfly 16, 8, 4, 2, 1 for every N, so a row's sum does not depend on the tile's size.
template <int N>
__device__ __forceinline__ float reduce_rows(float (&v)[N]) {
  const int lane = threadIdx.x & 31;
  int o = 16;
#pragma unroll
  for (int n = N / 2; n >= 1; n /= 2, o /= 2) {
    const bool hi = lane & o;
#pragma unroll
    for (int i = 0; i < n; ++i) {
      const float send = hi ? v[i] : v[i + n];
      const float keep = hi ? v[i + n] : v[i];
      v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
    }
  }
  float r = v[0];
#pragma unroll
  for (int q = 32 / N / 2; q >= 1; q /= 2) r += __shfl_xor_sync(0xffffffffu, r, q);
  return r;
}

// 16-byte global load (zero when !pred) and store.
__device__ __forceinline__ uint4 ldg_v4(const void* p, bool pred) {
  uint4 v;
  asm volatile(
      "{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %5, 0;\n\tmov.b32 %0, 0;\n\tmov.b32 %1, 0;\n\tmov.b32 %2, 0;\n\t"
      "mov.b32 %3, 0;\n\t@q ld.global.v4.b32 {%0, %1, %2, %3}, [%4];\n\t}"
      : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
      : "l"(p), "r"((uint32_t)pred)
      : "memory");
  return v;
}
__device__ __forceinline__ void stg_v4(void* p, uint4 v) {
  asm volatile("st.global.v4.b32 [%0], {%1, %2, %3, %4};" ::"l"(p), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}

__device__ __forceinline__ int nkb_of(int K) { return (K + KBLK - 1) / KBLK; }
__device__ __forceinline__ int nmc_of(int N) { return (N + MCH - 1) / MCH; }

// Slot of the split at (mask word w, bit) of a tile row, in the row's sorted split order:
// the splits in earlier words plus those below `bit` in word w (O(1), no search).
template <class SM>
__device__ __forceinline__ int split_slot(const SM* sm, int row, int w, int bit) {
  return (int)sm->wfirst[w][row] + __popc(sm->smask[w][row] & ((1u << bit) - 1u));
}

// ------------------------------------------------------------------------------------------
// The kernel
// ------------------------------------------------------------------------------------------
// MODE 0: bound only; MODE 1: bound and gradient (adjoint pass); MODE 2: as MODE 1 with dlb/dalpha
// stored in BF16 (the optimiser's own gradient buffer).  TR: rows per tile (16, 32 or 64).
//
// Contractions of a tile, in the order the TMA and MMA warps run them: backward layers L-1 .. 2;
// the concretisation (backward layer 1) interleaved with forward layer 1, whose operand x* the
// concretisation's epilogue writes chunk by chunk; forward layers 2 .. L-1.
template <int MODE, int TR>
__global__ void __launch_bounds__(NTHREADS, 1) k_fused(const __grid_constant__ Maps maps, const Args a) {
  using SM = Smem<TR>;
  constexpr int SLOT_BYTES = TR * 128;   // one K block of a slot
  constexpr int RW = TR / 4;             // rows of an epilogue warp
  constexpr int RS = RW < 8 ? RW : 8;    // rows per accumulator load
  constexpr int ACC_COLS = (NACC + (MODE >= 1 ? NFACC : 0)) * TR;
  constexpr int TMEM_COLS = ACC_COLS <= 64 ? 64 : ACC_COLS <= 128 ? 128 : ACC_COLS <= 256 ? 256 : 512;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  // pointer arithmetic on the shared array (not through an integer) keeps the shared address
  // space visible to the compiler, so accesses through `sm` are shared loads/stores
  const uint32_t pad = (1024u - (su32(smem_raw) & 1023u)) & 1023u;
  SM* sm = reinterpret_cast<SM*>(smem_raw + pad);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int n_tiles = a.n_tiles ? *a.n_tiles : a.tiles;

  if (threadIdx.x == 0) {
    for (int i = 0; i < NSLOT; ++i) {
      mbar_init(&sm->act_full[i], NEPI);
      mbar_init(&sm->act_empty[i], 1);
    }
    for (int i = 0; i < NSTAGE; ++i) {
      mbar_init(&sm->w_full[i], 1);
      mbar_init(&sm->w_empty[i], 1);
    }
    for (int i = 0; i < NACC; ++i) {
      mbar_init(&sm->acc_full[i], 1);
      mbar_init(&sm->acc_empty[i], NEPI);
    }
    mbar_init(&sm->facc_full, 1);
    mbar_init(&sm->epi, NEPI);
    mbar_init(&sm->done, 1);
    sm->abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == MMA_WARP) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(&sm->tmem_base)),
                 "n"(TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = sm->tmem_base;

  // The TMA and the MMA warp run their loops as whole warps (every lane takes the same waits and
  // branches) and one lane issues.  What bounds the MMA warp is its own instructions: with one K
  // block per wait and commit and a one-lane branch a 256-deep chunk of 16 MMAs took 1.7 us,
  // whatever the weight ring's depth (now 0.65).  The rest of a 64-row tile's time (118 -> 107 us
  // alone on its SM, 784-256x6-10) is its epilogues: 1.0-1.3 us a chunk backward, 2.2-2.6 forward.
  if (warp == TMA_WARP) {
    // ---------------------------------------------------------------- TMA producer
    uint32_t wseq = 0, st = 0, ph = 1;
    bool ok = true;
    // K pair kp of M chunk mc of a layer's weights
    auto put = [&](const CUtensorMap* map, uint32_t bytes, int mc, int kp, int nkb) -> bool {
      if (!mbar_wait_all(&sm->w_empty[st], ph, sm, a.status)) return false;
      if (lane == 0) {
        const bool two = 2 * kp + 1 < nkb;
        mbar_expect_tx(&sm->w_full[st], two ? 2 * bytes : bytes);
        tma_load_2d(sm->w[st], map, 2 * kp * KBLK, mc * MCH, &sm->w_full[st]);
        if (two) tma_load_2d(sm->w[st] + STAGE_BYTES, map, (2 * kp + 1) * KBLK, mc * MCH, &sm->w_full[st]);
      }
      ++wseq;
      if (++st == NSTAGE) st = 0, ph ^= 1;
      return true;
    };
    // all chunks of a layer with a resident operand
    auto layer = [&](bool fwd, int i) -> bool {
      const CUtensorMap* map = fwd ? &maps.fwd[i] : &maps.bwd[i];
      const uint32_t bytes = (uint32_t)(fwd ? a.box_fwd[i] : a.box_bwd[i]) * 128u;
      const int nmc = nmc_of(a.d[fwd ? i : i - 1]), nkb = nkb_of(a.d[fwd ? i - 1 : i]), nkp = (nkb + 1) / 2;
      for (int mc = 0; mc < nmc; ++mc)
        for (int kp = 0; kp < nkp; ++kp)
          if (!put(map, bytes, mc, kp, nkb)) return false;
      return true;
    };
    for (int tile = blockIdx.x; tile < n_tiles && ok; tile += gridDim.x) {
      for (int i = a.L - 1; i >= 2 && ok; --i) ok = layer(false, i);
      const uint32_t cb = (uint32_t)a.box_bwd[1] * 128u, fb = (uint32_t)a.box_fwd[1] * 128u;
      const int ncx = nmc_of(a.d[0]), nkb1 = nkb_of(a.d[1]), nkp1 = (nkb1 + 1) / 2;
      const int nkbx = nkb_of(a.d[0]), nmc1 = nmc_of(a.d[1]);
      for (int m = 0; m < ncx + (MODE >= 1 ? XLAG : 0) && ok; ++m) {
        if (m < ncx)
          for (int kp = 0; kp < nkp1 && ok; ++kp) ok = put(&maps.bwd[1], cb, m, kp, nkb1);
        if (MODE >= 1 && m >= XLAG)
          for (int mc = 0; mc < nmc1 && ok; ++mc) ok = put(&maps.fwd[1], fb, mc, m - XLAG, nkbx);
      }
      if (MODE >= 1)
        for (int i = 2; i <= a.L - 1 && ok; ++i) ok = layer(true, i);
    }
    if (!ok && lane == 0) {
      // wait (bounded) for the copies still in flight before the CTA may exit
      for (uint32_t s = (wseq > NSTAGE ? wseq - NSTAGE : 0); s < wseq; ++s) {
        long long t0 = clock64();
        while (!mbar_try(&sm->w_full[s % NSTAGE], (s / NSTAGE) & 1) && clock64() - t0 < 200000000LL) {
        }
      }
    }
  } else if (warp == MMA_WARP) {
    // ---------------------------------------------------------------- MMA issuer
    // (st, wph): the weight stage read next and the parity of its full barrier; half, fpar: the
    // slots of the operand read next, and per slot the parity of its full barrier; (buf, cph): the
    // accumulator filled next and the parity of its empty barrier
    uint32_t st = 0, wph = 0, half = 0, fpar = 0, buf = 0, cph = 1;
    const uint32_t w0 = sdesc_lo(su32(sm->w[0])), a0 = sdesc_lo(su32(sm->act[0]));
    const uint32_t b_wempty = su32(&sm->w_empty[0]), b_aempty = su32(&sm->act_empty[0]), b_acc = su32(&sm->acc_full[0]);
    constexpr uint32_t WSTEP = 2 * STAGE_BYTES >> 4, ASTEP = 2 * SLOT_BYTES >> 4;
    constexpr uint32_t idesc = idesc_bf16(TR);
    bool ok = true;
    // one K pair (or its first block) of a chunk: weights of stage st, activations of slot s
    auto pair = [&](uint32_t dt, uint32_t s, bool first, bool two) -> bool {
      if (!mbar_wait_all(&sm->w_full[st], wph, sm, a.status)) return false;
      tc_fence_after();
      umma_kpair<(STAGE_BYTES >> 4), (SLOT_BYTES >> 4)>(dt, w0 + st * WSTEP, a0 + s * ASTEP, idesc, first ? 0u : 1u,
                                                        two ? 1u : 0u, b_wempty + 8 * st);
      if (++st == NSTAGE) st = 0, wph ^= 1;
      return true;
    };
    // chunk mc of nmc of a contraction with a resident operand (slots half, half + 1) of nkb K blocks
    auto chunk = [&](int mc, int nmc, int nkb) -> bool {
      const bool last = mc == nmc - 1;
      if (!mbar_wait_all(&sm->acc_empty[buf], cph, sm, a.status)) return false;
      tc_fence_after();
      const uint32_t dt = tmem + buf * TR;
      if (mc == 0 && !mbar_wait_all(&sm->act_full[half], (fpar >> half) & 1, sm, a.status)) return false;
      if (!pair(dt, half, true, nkb > 1)) return false;
      if (last) umma_commit_warp(b_aempty + 8 * half);
      if (nkb > 2) {
        if (mc == 0 && !mbar_wait_all(&sm->act_full[half + 1], (fpar >> (half + 1)) & 1, sm, a.status)) return false;
        if (!pair(dt, half + 1, false, nkb > 3)) return false;
        if (last) umma_commit_warp(b_aempty + 8 * (half + 1));
      }
      umma_commit_warp(b_acc + 8 * buf);
      if (++buf == NACC) buf = 0, cph ^= 1;
      if (last) {
        fpar ^= (nkb > 2 ? 3u : 1u) << half;
        half ^= 2;
      }
      return true;
    };
    for (int tile = blockIdx.x; tile < n_tiles && ok; tile += gridDim.x) {
      for (int i = a.L - 1; i >= 2 && ok; --i) {
        const int nmc = nmc_of(a.d[i - 1]), nkb = nkb_of(a.d[i]);
        for (int mc = 0; mc < nmc && ok; ++mc) ok = chunk(mc, nmc, nkb);
      }
      // the concretisation's chunks, and forward layer 1 over the x* pairs they yield, XLAG behind:
      // the chunk that waits for the accumulator of chunk e finds x* pair e written.  x* takes the
      // half that Lambda^(1) does not, one slot after the other.
      const int ncx = nmc_of(a.d[0]), nkb1 = nkb_of(a.d[1]);
      const int nkbx = nkb_of(a.d[0]), nmc1 = nmc_of(a.d[1]);
      const uint32_t xhalf = half ^ 2;
      for (int m = 0; m < ncx + (MODE >= 1 ? XLAG : 0) && ok; ++m) {
        if (m < ncx && !(ok = chunk(m, ncx, nkb1))) break;
        if (MODE == 0 || m < XLAG) continue;
        const int e = m - XLAG;
        const uint32_t s = xhalf + (uint32_t)(e & 1);
        if (!(ok = mbar_wait_all(&sm->act_full[s], (fpar >> s) & 1, sm, a.status))) break;
        for (int mc = 0; mc < nmc1 && ok; ++mc)
          ok = pair(tmem + (uint32_t)((NACC + mc) * TR), s, e == 0, 2 * e + 1 < nkbx);
        if (!ok) break;
        umma_commit_warp(b_aempty + 8 * s);
        fpar ^= 1u << s;
      }
      if (!ok) break;
      if (MODE >= 1) {
        umma_commit_warp(su32(&sm->facc_full));
        half = xhalf ^ 2;
        for (int i = 2; i <= a.L - 1 && ok; ++i) {
          const int nmc = nmc_of(a.d[i]), nkb = nkb_of(a.d[i - 1]);
          for (int mc = 0; mc < nmc && ok; ++mc) ok = chunk(mc, nmc, nkb);
        }
      }
    }
    __syncwarp();
    umma_commit_warp(su32(&sm->done));
    mbar_wait_all(&sm->done, 0, sm, a.status);
  } else {
    // ---------------------------------------------------------------- epilogue (warps 0..15)
    const int q = warp & 3;          // TMEM lane quadrant: neurons 32q..32q+31 of an M chunk
    const int cg = warp >> 2;        // column group: tile rows RW cg .. RW cg + RW - 1
    const int r0 = RW * cg;          // first tile row of this thread
    const int etid = threadIdx.x;    // 0..511
    // the operand written next (its slots' first), per slot the parity of its empty barrier, the
    // accumulator read next
    uint32_t half = 0, epar = 0, accseq = 0, eseq = 0, fph = 0;
    bool ok = true;

    for (int tile = blockIdx.x; tile < n_tiles && ok; tile += gridDim.x) {
      // Every row of a tile belongs to one property (the rows are grouped by property before
      // the launch); slots past the property's last row are empty.
      const int p = a.n_tiles ? a.tile_prop[tile] : 0;
      // ---------------- tile set-up, step 1: per-row scalars (one thread per row)
      if (warp < (TR + 31) / 32) {
        const int row = etid;
        int v = 0, r = -1;
        if (row < TR) {
          r = a.n_tiles ? a.rowmap[(size_t)tile * TR + row] : tile * TR + row;
          v = r >= 0 && r < a.R && p >= 0 && p < a.P;
          if (!a.n_tiles && v && a.bt.prop_of[r / a.K] != 0) {   // (the planner checks the others)
            atomicCAS(a.status, 0, BCROWN_ERR_ARG);
            v = 0;
          }
          int k = 0, cnt = 0, off = 0;
          long long ab = 0, bb = 0;
          if (v) {
            const int b = r / a.K;
            k = r - b * a.K;
            cnt = a.bt.split_cnt[b];
            off = a.bt.split_off[b];
            const long long ao = a.bt.alpha_off[b];
            const int U = a.tb.U[p];
            ab = ao + (long long)k * U;
            bb = (long long)off * a.K + (long long)k * cnt;
            // every alpha of the row must lie in the array: then no per-element check is needed
            if (cnt < 0 || cnt > BCROWN_MAX_SPLITS || off < 0 || ab < 0 || ab + U > a.n_alpha) {
              atomicCAS(a.status, 0, BCROWN_ERR_ARG);
              v = 0;
            }
          }
          sm->valid[row] = v;
          sm->rowid[row] = v ? r : -1;
          sm->spec[row] = v ? k : 0;
          sm->scnt[row] = v ? cnt : 0;
          sm->soff[row] = off;
          sm->abase[row] = v ? ab : 0;
          sm->bbase[row] = v ? bb : 0;
          sm->part[0][row] = sm->part[1][row] = sm->part[2][row] = sm->part[3][row] = 0.f;
        }
        const unsigned vb = __ballot_sync(0xffffffffu, v != 0);
        if (lane == 0) reinterpret_cast<uint32_t*>(&sm->vrows)[warp] = vb;
        if (TR < 64 && lane == 0) reinterpret_cast<uint32_t*>(&sm->vrows)[1] = 0u;
      }
      const int pp = (p >= 0 && p < a.P) ? p : 0;
      {
        // the property's per-neuron tables
        // all loads first, then the stores (3 neurons per thread at most)
        constexpr int NT = (MAX_H + NEPI * 32 - 1) / (NEPI * 32);
        int cd[NT], rk[NT];
        float sl[NT], ic[NT];
#pragma unroll
        for (int u = 0; u < NT; ++u) {
          const int nn = etid + u * NEPI * 32;
          const size_t g = (size_t)pp * a.H + nn;
          const bool in = nn < a.H;
          cd[u] = in ? a.tb.code[g] : 0;
          rk[u] = in ? a.tb.rank[g] : 0;
          sl[u] = in ? a.tb.slope[g] : 0.f;
          ic[u] = in ? a.tb.icpt[g] : 0.f;
        }
#pragma unroll
        for (int u = 0; u < NT; ++u) {
          const int nn = etid + u * NEPI * 32;
          if (nn < a.H) {
            sm->tcode[nn] = ((uint32_t)cd[u] << 16) | (uint32_t)(rk[u] < 0 ? 0xFFFF : (rk[u] & 0xFFFF));
            sm->tslope[nn] = sl[u];
            sm->ticpt[nn] = ic[u];
          }
        }
      }
      for (int x = etid; x < a.mask_words * TR; x += NEPI * 32) (&sm->smask[0][0])[x] = 0u;
      if (etid < a.mask_words) sm->wrows[etid] = 0ull;
      if (!epi_sync(sm, eseq, a.status)) {
        ok = false;
        break;
      }
      // ---------------- step 2: split masks (8 threads per row) and the splits' beta S
      const int srow = etid >> 3, e0 = etid & 7;
      const bool has_row = srow < TR;   // the same for a whole warp
      int ent[BCROWN_MAX_SPLITS / 8];   // this thread's split entries: mask word << 5 | bit, or -1
      float bv[BCROWN_MAX_SPLITS / 8];  // and their beta (loaded now, stored in step 4)
      if (has_row) {
        const int cnt = sm->scnt[srow], off = sm->soff[srow];
#pragma unroll
        for (int m = 0; m < BCROWN_MAX_SPLITS / 8; ++m) {
          const long long bi = sm->bbase[srow] + e0 + 8 * m;
          bv[m] = ldg_f32(a.beta + bi, e0 + 8 * m < cnt && bi >= 0 && bi < a.n_beta);
        }
#pragma unroll
        for (int m = 0; m < BCROWN_MAX_SPLITS / 8; ++m) {
          const int e = e0 + 8 * m;
          ent[m] = -1;
          if (e < cnt) {
            const int ly = a.bt.split_layer[off + e];
            const int j = (int)a.bt.split_idx[off + e];
            const int s = a.bt.split_sign[off + e];
            if (ly < 1 || ly > a.L - 1 || j < 0 || j >= a.d[ly] || (s != 1 && s != -1)) {
              atomicCAS(a.status, 0, BCROWN_ERR_ARG);
            } else {
              const int wd = a.woff[ly] + (j >> 5);
              atomicOr(&sm->smask[wd][srow], 1u << (j & 31));
              ent[m] = (wd << 5) | (j & 31);
              bv[m] = fmaxf(bv[m], 0.f) * (float)s;
            }
          }
        }
      }
      if (!epi_sync(sm, eseq, a.status)) {
        ok = false;
        break;
      }
      // ---------------- step 3: per-row split counts before each mask word (a prefix over the
      // row's 8 threads, 6 words each) and the rows with a split in each word (shared atomics)
      if (has_row) {
        const int part = e0;
        constexpr int WPT = MAX_MASK_WORDS / 8;
        int cw[WPT];
        int loc = 0;
#pragma unroll
        for (int u = 0; u < WPT; ++u) {
          const int w = part * WPT + u;
          const uint32_t m = w < a.mask_words ? sm->smask[w][srow] : 0u;
          cw[u] = __popc(m);
          loc += cw[u];
          if (m) atomicOr(&sm->wrows[w], 1ull << srow);
        }
        int incl = loc;
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) {
          const int y = __shfl_up_sync(0xffffffffu, incl, o, 8);
          if (part >= o) incl += y;
        }
        int run = incl - loc;
#pragma unroll
        for (int u = 0; u < WPT; ++u) {
          const int w = part * WPT + u;
          if (w < a.mask_words) sm->wfirst[w][srow] = (uint8_t)run;
          run += cw[u];
        }
      }
      if (!epi_sync(sm, eseq, a.status)) {
        ok = false;
        break;
      }
      // ---------------- step 4: each split's slot in (word, bit) order, its list position and beta S
      if (has_row) {
#pragma unroll
        for (int m = 0; m < BCROWN_MAX_SPLITS / 8; ++m) {
          if (ent[m] >= 0) {
            const int ks = split_slot(sm, srow, ent[m] >> 5, ent[m] & 31);
            sm->sorig[srow][ks] = (uint8_t)(e0 + 8 * m);
            sm->sbeta[srow][ks] = bv[m];
          }
        }
      }
      if (!epi_sync(sm, eseq, a.status)) {
        ok = false;
        break;
      }
      // rows of this thread that take part (bit c: tile row r0 + c); empty rows have all-zero
      // operands, so they only need their global loads and stores masked
      constexpr uint32_t ALL = RW == 32 ? ~0u : (1u << RW) - 1u;
      const uint32_t vbits = (uint32_t)(sm->vrows >> r0) & ALL;

      // alpha (or 0 where !pred) of the thread's RW rows at rank: p = a.alpha + rank
      auto load_alpha = [&](const float* pa, bool pred, float (&al)[RW]) {
#pragma unroll
        for (int c = 0; c < RW; c += 4) {
          const longlong2 b0 = *reinterpret_cast<const longlong2*>(&sm->abase[r0 + c]);
          const longlong2 b1 = *reinterpret_cast<const longlong2*>(&sm->abase[r0 + c + 2]);
          const uint32_t v4 = (vbits >> c) & 15u;
          if (v4 == 15u) {
            ldg4_f32(pa + b0.x, pa + b0.y, pa + b1.x, pa + b1.y, pred, &al[c]);
          } else {
            al[c] = ldg_f32(pa + b0.x, pred && (v4 & 1u));
            al[c + 1] = ldg_f32(pa + b0.y, pred && (v4 & 2u));
            al[c + 2] = ldg_f32(pa + b1.x, pred && (v4 & 4u));
            al[c + 3] = ldg_f32(pa + b1.y, pred && (v4 & 8u));
          }
        }
      };

      // per-thread lb partial sums of its rows over the lanes' neurons (whole backward pass)
      float racc[RW];
#pragma unroll
      for (int c = 0; c < RW; ++c) racc[c] = 0.f;

      // ---------------- backward pass: A^(i-1) = Lambda^(i) W^(i) from the accumulator, relaxed
      // into the next operand Lambda^(i-1).  i = L is the top: A^(L-1) = Wbar (no contraction).
      for (int i = a.L; i >= 2 && ok; --i) {
        const bool top = (i == a.L);
        const int N = a.d[i - 1];
        const int nmc = nmc_of(N);
        const int li = i - 1;
        const int nkb_next = nkb_of(N);
        for (int mc = 0; mc < nmc && ok; ++mc) {
          const int buf = accseq % NACC;
          const int j = mc * MCH + 32 * q + lane;   // output neuron of this lane
          const bool jin = j < N;
          // ---- relaxation of layer i-1 (Lemma 2.1 / Eq. definition_D, split override of Eq. 3)
          // D = 1 active, 0 inactive; unstable: alpha where A >= 0, the chord slope (+ intercept
          // lambda) where A < 0; a split neuron takes D = 1 or 0 and adds beta S.
          const long long n = a.hoff[li] + j;
          int code = CODE_INACTIVE, rank = 0;
          float dneg = 0.f, lneg = 0.f;
          const float bj = ldg_f32(a.bias[li] + j, jin);
          if (jin) {
            const uint32_t t = sm->tcode[n];
            code = (int)(t >> 16);
            rank = (int)(t & 0xFFFF);
            dneg = code == CODE_ACTIVE ? 1.f : (code == CODE_UNSTABLE ? sm->tslope[n] : 0.f);
            lneg = code == CODE_UNSTABLE ? sm->ticpt[n] : 0.f;
          }
          const bool unst = code == CODE_UNSTABLE;
          const float apos = code == CODE_ACTIVE ? 1.f : 0.f;
          const int kb = (mc * MCH + 32 * q) / KBLK;   // this warp's K block of the next operand
          const bool writer = kb < nkb_next;           // (the pair's second block may lie past the end)
          const uint32_t slot = half + (uint32_t)mc;   // chunk mc is K pair mc of the next operand
          // split bits of the warp's 32 neurons (none when they all lie past the layer's end)
          const int wd = a.woff[li] + ((mc * MCH + 32 * q) >> 5);
          const uint32_t bit = 1u << lane;
          const uint32_t rbits = mc * MCH + 32 * q < N ? (uint32_t)(sm->wrows[wd] >> r0) & ALL : 0u;
          // alpha of the rows, issued before waiting for the accumulator
          float al[RW];
          load_alpha(a.alpha + rank, unst, al);
          // byte offset of (row r0 + RS h + c8, k = j % 64) in the slot's block; row & 7 is known
          // per c8 but for tiles of 16 rows, whose warps start on a multiple of 4
          const int kk = j & (KBLK - 1);
          uint8_t* aslot = sm->act[slot] + (kb & 1) * SLOT_BYTES + r0 * 128 + ((kk & 7) << 1);
          const uint32_t kx = ((uint32_t)(kk >> 3) ^ (uint32_t)(RS < 8 ? r0 & 7 : 0)) << 4;
          __nv_bfloat16* st_p = MODE >= 1 ? a.stash + ((size_t)tile * a.H + n) * TR + r0 : nullptr;
          // rows r0 + RS h .. of A^(i-1)_j: relaxation, lb terms, operand and stash
          auto relax8 = [&](const int h, const float (&v)[RS]) {
#pragma unroll
            for (int c8 = 0; c8 < RS; ++c8) {
              const int c = RS * h + c8;
              const int row = r0 + c;
              const float av = v[c8];
              const bool pos = av >= 0.f;
              float D = pos ? __saturatef(al[c] + apos) : dneg;
              float lm = pos ? 0.f : lneg;
              float bs = 0.f;
              if ((rbits >> c) & 1u) {
                if (sm->smask[wd][row] & bit) {
                  bs = sm->sbeta[row][split_slot(sm, row, wd, lane)];
                  D = signbit(bs) ? 1.f : 0.f;
                  lm = 0.f;
                }
              }
              const float L = fmaf(av, D, bs);
              racc[c] = fmaf(L, bj, fmaf(av, lm, racc[c]));
              if (writer)
                *reinterpret_cast<__nv_bfloat16*>(aslot + (RS * h + c8) * 128 + (kx ^ (uint32_t)(c8 << 4))) =
                    __float2bfloat16_rn(L);
            }
            if constexpr (MODE >= 1) {
              // A^(i-1) of the rows for the adjoint pass: one store per lane
              if (jin) {
                uint32_t pk[RS / 2];
#pragma unroll
                for (int e = 0; e < RS; e += 2) {
                  __nv_bfloat162 v2 = __floats2bfloat162_rn(v[e], v[e + 1]);
                  pk[e >> 1] = *reinterpret_cast<uint32_t*>(&v2);
                }
                if constexpr (RS == 8) stg_v4(st_p + RS * h, make_uint4(pk[0], pk[1], pk[2], pk[3]));
                else *reinterpret_cast<uint2*>(st_p) = make_uint2(pk[0], pk[1]);
              }
            }
          };
          if (!top) {
            if (!mbar_wait_warp(&sm->acc_full[buf], (accseq / NACC) & 1, sm, a.status)) {
              ok = false;
              break;
            }
            tc_fence_after();
          }
          if (!mbar_wait_warp(&sm->act_empty[slot], ((epar >> slot) & 1) ^ 1, sm, a.status)) {
            ok = false;
            break;
          }
          const uint32_t tbase = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(buf * TR + r0);
          if (top) {
#pragma unroll
            for (int h = 0; h < RW / RS; ++h) {
              // A^(L-1) = Wbar rows of the rows' specifications
              float v[RS];
#pragma unroll
              for (int c8 = 0; c8 < RS; ++c8) {
                const int c = RS * h + c8;
                v[c8] = ldg_f32(a.Wbar + (size_t)sm->spec[r0 + c] * N + j, jin && ((vbits >> c) & 1u));
              }
              relax8(h, v);
            }
          } else {
            // RS rows, then the next RS: the second load runs under the first rows' work
            uint32_t u[RW / RS][RS];
            tmem_ld_issue(tbase, u[0]);
#pragma unroll
            for (int h = 0; h < RW / RS; ++h) {
              tmem_wait(u[h]);
              if (h + 1 < RW / RS) {
                tmem_ld_issue(tbase + RS * (h + 1), u[h + 1 < RW / RS ? h + 1 : h]);
              } else {
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbar_arrive(&sm->acc_empty[buf]);
                ++accseq;
              }
              float v[RS];
#pragma unroll
              for (int e = 0; e < RS; ++e) v[e] = __uint_as_float(u[h][e]);
              relax8(h, v);
            }
          }
          // each K pair is complete once all warps arrived
          fence_proxy_async();
          __syncwarp();
          if (lane == 0) mbar_arrive(&sm->act_full[slot]);
          epar ^= 1u << slot;
        }
        half ^= 2;
      }
      if (!ok) break;

      // ---------------- concretisation: lb += sum_m min(A_m x_lo_m, A_m x_hi_m) (Eq. beta_crown_lp)
      // and, for the adjoint, x* (the point of the box that minimises A^(0) x: x_lo where A^(0) >= 0,
      // else x_hi) as the operand of forward layer 1, chunk e = K pair e in slot e & 1 of the half
      // that Lambda^(1) does not hold
      {
        const int N = a.d[0];
        const int ncx = nmc_of(N);
        for (int e = 0; e < ncx && ok; ++e) {
          const int buf = accseq % NACC;
          const int j = e * MCH + 32 * q + lane;
          const bool jin = j < N;
          const float uxl = ldg_f32(a.x_lo + (size_t)pp * N + j, jin), uxh = ldg_f32(a.x_hi + (size_t)pp * N + j, jin);
          const uint32_t slot = half + (uint32_t)(e & 1);
          const int kk = j & (KBLK - 1);
          uint8_t* aslot = sm->act[slot] + ((j / KBLK) & 1) * SLOT_BYTES + r0 * 128 + ((kk & 7) << 1);
          const uint32_t kx = ((uint32_t)(kk >> 3) ^ (uint32_t)(RS < 8 ? r0 & 7 : 0)) << 4;
          const uint32_t tbase = tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(buf * TR + r0);
          if (!mbar_wait_warp(&sm->acc_full[buf], (accseq / NACC) & 1, sm, a.status)) {
            ok = false;
            break;
          }
          tc_fence_after();
          uint32_t u[RW / RS][RS];
#pragma unroll
          for (int h = 0; h < RW / RS; ++h) tmem_ld_issue(tbase + RS * h, u[h]);
#pragma unroll
          for (int h = 0; h < RW / RS; ++h) tmem_wait(u[h]);
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(&sm->acc_empty[buf]);
          ++accseq;
          if (MODE >= 1 && !mbar_wait_warp(&sm->act_empty[slot], ((epar >> slot) & 1) ^ 1, sm, a.status)) {
            ok = false;
            break;
          }
          const __nv_bfloat16 bl = __float2bfloat16_rn(uxl), bh = __float2bfloat16_rn(uxh);
#pragma unroll
          for (int c = 0; c < RW; ++c) {
            const float av = __uint_as_float(u[c / RS][c % RS]);
            racc[c] += fminf(av * uxl, av * uxh);
            if constexpr (MODE >= 1) {
              const bool rin = (vbits >> c) & 1u;
              *reinterpret_cast<__nv_bfloat16*>(aslot + c * 128 + (kx ^ (uint32_t)((c % RS) << 4))) =
                  rin ? (av >= 0.f ? bl : bh) : __float2bfloat16_rn(0.f);
            }
          }
          if constexpr (MODE >= 1) {
            fence_proxy_async();
            __syncwarp();
            if (lane == 0) mbar_arrive(&sm->act_full[slot]);
            epar ^= 1u << slot;
          }
        }
        if (MODE >= 1) half ^= 2;
      }
      if (!ok) break;

      // ---------------- lb of each row: reduce the lanes' partial sums, then the quadrants'
      {
        const float rs = reduce_rows(racc);
        if (lane % (32 / RW) == 0) atomicAdd(&sm->part[q][r0 + lane / (32 / RW)], rs);
      }
      if (!epi_sync(sm, eseq, a.status)) {
        ok = false;
        break;
      }
      if (etid < TR && sm->valid[etid]) {
        const int row = etid;
        float lbv = a.bbar[sm->spec[row]] + ((sm->part[0][row] + sm->part[1][row]) + (sm->part[2][row] + sm->part[3][row]));
        if (!isfinite(lbv)) {
          atomicCAS(a.status, 0, BCROWN_ERR_NONFINITE);
          lbv = -INFINITY;
        }
        a.lb[sm->rowid[row]] = lbv;
      }
      if constexpr (MODE >= 1) {
        // ---------------- adjoint: zhat^(i) = W^(i) h^(i-1) + b^(i); dalpha = A zhat (unstable, unsplit,
        // A >= 0), dbeta = S zhat; h^(i) = D zhat + lambda is the next forward operand
        for (int i = 1; i <= a.L - 1 && ok; ++i) {
          const int N = a.d[i];
          const int nmc = nmc_of(N);
          const int nkb_next = (i + 1 <= a.L - 1) ? nkb_of(N) : 0;
          for (int mc = 0; mc < nmc && ok; ++mc) {
            const int buf = accseq % NACC;
            const int j = mc * MCH + 32 * q + lane;
            const bool jin = j < N;
            const long long n = a.hoff[i] + j;
            int code = CODE_INACTIVE, rank = 0;
            float dneg = 0.f, lneg = 0.f;
            const float bj = ldg_f32(a.bias[i] + j, jin);
            if (jin) {
              const uint32_t t = sm->tcode[n];
              code = (int)(t >> 16);
              rank = (int)(t & 0xFFFF);
              dneg = code == CODE_ACTIVE ? 1.f : (code == CODE_UNSTABLE ? sm->tslope[n] : 0.f);
              lneg = code == CODE_UNSTABLE ? sm->ticpt[n] : 0.f;
            }
            const bool unst = code == CODE_UNSTABLE;
            const float apos = code == CODE_ACTIVE ? 1.f : 0.f;
            const int kb = (mc * MCH + 32 * q) / KBLK;
            const bool writer = kb < nkb_next;
            const bool pwriter = nkb_next > 0;
            const uint32_t slot = half + (uint32_t)mc;
            const int wd = a.woff[i] + ((mc * MCH + 32 * q) >> 5);
            const uint32_t bit = 1u << lane;
            const uint32_t rbits = mc * MCH + 32 * q < N ? (uint32_t)(sm->wrows[wd] >> r0) & ALL : 0u;
            // A^(i) of the rows and alpha, issued before the accumulator wait
            const __nv_bfloat16* sp = a.stash + ((size_t)tile * a.H + n) * TR + r0;
            uint32_t sw[RW / 2];
            if constexpr (RS == 8) {
#pragma unroll
              for (int h = 0; h < RW / RS; ++h) {
                const uint4 x = ldg_v4(sp + 8 * h, jin);
                sw[4 * h] = x.x, sw[4 * h + 1] = x.y, sw[4 * h + 2] = x.z, sw[4 * h + 3] = x.w;
              }
            } else {
              const uint2 x = jin ? *reinterpret_cast<const uint2*>(sp) : make_uint2(0u, 0u);
              sw[0] = x.x, sw[1] = x.y;
            }
            float al[RW];
            load_alpha(a.alpha + rank, unst, al);
            // layer 1 accumulates apart from the ring (all its chunks over the x* stream)
            if (!mbar_wait_warp(i == 1 ? &sm->facc_full : &sm->acc_full[buf], i == 1 ? fph : (accseq / NACC) & 1, sm,
                                a.status)) {
              ok = false;
              break;
            }
            tc_fence_after();
            if (pwriter && !mbar_wait_warp(&sm->act_empty[slot], ((epar >> slot) & 1) ^ 1, sm, a.status)) {
              ok = false;
              break;
            }
            const int kk = j & (KBLK - 1);
            uint8_t* aslot = sm->act[slot] + (kb & 1) * SLOT_BYTES + r0 * 128 + ((kk & 7) << 1);
            const uint32_t kx = ((uint32_t)(kk >> 3) ^ (uint32_t)(RS < 8 ? r0 & 7 : 0)) << 4;
            const uint32_t tbase =
                tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)((i == 1 ? NACC + mc : buf) * TR + r0);
            // rows r0 + RS h ..: zhat, gradients, next operand
            auto fwd8 = [&](const int h, const uint32_t (&u)[RS]) {
#pragma unroll
              for (int c8 = 0; c8 < RS; ++c8) {
                const int c = RS * h + c8;
                const int row = r0 + c;
                const bool rin = (vbits >> c) & 1u;
                const uint32_t w = sw[c >> 1];
                const float A = __uint_as_float((c & 1) ? (w & 0xFFFF0000u) : (w << 16));
                const float z = __uint_as_float(u[c8]) + bj;
                const bool pos = A >= 0.f;
                float D = pos ? __saturatef(al[c] + apos) : dneg;
                float lm = pos ? 0.f : lneg;
                float g = pos ? A * z : 0.f;
                if ((rbits >> c) & 1u) {
                  if (sm->smask[wd][row] & bit) {
                    const int ks = split_slot(sm, row, wd, lane);
                    const bool neg = signbit(sm->sbeta[row][ks]);   // S = -1: z >= 0
                    D = neg ? 1.f : 0.f;
                    lm = 0.f;
                    g = 0.f;
                    const long long bi = sm->bbase[row] + sm->sorig[row][ks];
                    if (bi < a.n_beta) a.dbeta[bi] = neg ? -z : z;
                  }
                }
                if (unst && rin) {
                  if constexpr (MODE == 2) (a.dalpha16 + rank)[sm->abase[row]] = __float2bfloat16_rn(g);
                  else (a.dalpha + rank)[sm->abase[row]] = g;
                }
                const float hv = rin ? fmaf(D, z, lm) : 0.f;
                if (writer)
                  *reinterpret_cast<__nv_bfloat16*>(aslot + (RS * h + c8) * 128 + (kx ^ (uint32_t)(c8 << 4))) =
                      __float2bfloat16_rn(hv);
              }
            };
            uint32_t u[RW / RS][RS];
            tmem_ld_issue(tbase, u[0]);
#pragma unroll
            for (int h = 0; h < RW / RS; ++h) {
              tmem_wait(u[h]);
              if (h + 1 < RW / RS) {
                tmem_ld_issue(tbase + RS * (h + 1), u[h + 1 < RW / RS ? h + 1 : h]);
              } else {
                tc_fence_before();
                __syncwarp();
                if (i != 1) {
                  if (lane == 0) mbar_arrive(&sm->acc_empty[buf]);
                  ++accseq;
                }
              }
              fwd8(h, u[h]);
            }
            if (pwriter) {
              fence_proxy_async();
              __syncwarp();
              if (lane == 0) mbar_arrive(&sm->act_full[slot]);
              epar ^= 1u << slot;
            }
          }
          if (nkb_next > 0) half ^= 2;
          if (i == 1) fph ^= 1;
        }
        if (ok && !epi_sync(sm, eseq, a.status)) ok = false;
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == MMA_WARP) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "n"(TMEM_COLS) : "memory");
  }
}

// ------------------------------------------------------------------------------------------
// Row planner: group the rows (subdomain, spec) by property into tiles of `tr` rows, so that the
// fused kernel stages one property's tables per tile.  Row results do not depend on the tile a
// row lands in (each row is one column of every contraction), so the order inside a property
// is free; it is taken from atomic counters.
// ------------------------------------------------------------------------------------------
__global__ void k_plan_count(int B, int P, const int32_t* __restrict__ prop_of, int* __restrict__ cnt, int* status) {
  for (int b = blockIdx.x * blockDim.x + threadIdx.x; b < B; b += gridDim.x * blockDim.x) {
    const int p = prop_of[b];
    if (p < 0 || p >= P) {
      atomicCAS(status, 0, BCROWN_ERR_ARG);
      continue;
    }
    atomicAdd(&cnt[p], 1);
  }
}

// Exclusive prefix sums over the properties of their subdomains and of their tiles (one block).
__global__ void __launch_bounds__(1024) k_plan_scan(int P, int K, int tr, const int* __restrict__ cnt, int* __restrict__ cursor,
                                                    int* __restrict__ sub_base, int* __restrict__ tile_base,
                                                    int* __restrict__ n_tiles) {
  __shared__ int ws[32], wt[32];
  __shared__ int run_s, run_t;
  if (threadIdx.x == 0) run_s = run_t = 0;
  __syncthreads();
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (int base = 0; base < P; base += blockDim.x) {
    const int p = base + threadIdx.x;
    const int c = p < P ? cnt[p] : 0;
    const int t = (int)(((long long)c * K + tr - 1) / tr);
    int is = c, it = t;   // inclusive scans within the warp
    for (int o = 1; o < 32; o <<= 1) {
      const int xs = __shfl_up_sync(0xffffffffu, is, o), xt = __shfl_up_sync(0xffffffffu, it, o);
      if (lane >= o) {
        is += xs;
        it += xt;
      }
    }
    if (lane == 31) {
      ws[w] = is;
      wt[w] = it;
    }
    __syncthreads();
    int os = run_s, ot = run_t;
    for (int q = 0; q < w; ++q) {
      os += ws[q];
      ot += wt[q];
    }
    if (p < P) {
      sub_base[p] = os + is - c;
      tile_base[p] = ot + it - t;
      cursor[p] = 0;
    }
    __syncthreads();
    if (threadIdx.x == blockDim.x - 1) {
      run_s = os + is;
      run_t = ot + it;
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    sub_base[P] = run_s;
    tile_base[P] = run_t;
    *n_tiles = run_t;
  }
}

__global__ void k_plan_scatter(int B, int P, const int32_t* __restrict__ prop_of, const int* __restrict__ sub_base,
                               int* __restrict__ cursor, int* __restrict__ perm) {
  for (int b = blockIdx.x * blockDim.x + threadIdx.x; b < B; b += gridDim.x * blockDim.x) {
    const int p = prop_of[b];
    if (p < 0 || p >= P) continue;
    perm[sub_base[p] + atomicAdd(&cursor[p], 1)] = b;
  }
}

// Slot s of tile t: the property whose tiles contain t, and the global row in that slot.
__global__ void k_plan_rows(int max_tiles, int K, int P, int tr, const int* __restrict__ n_tiles,
                            const int* __restrict__ tile_base, const int* __restrict__ sub_base,
                            const int* __restrict__ perm, int* __restrict__ tile_prop, int* __restrict__ rowmap) {
  const long long id = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (id >= (long long)max_tiles * tr) return;
  const int t = (int)(id / tr), sl = (int)(id - (long long)t * tr);
  if (t >= *n_tiles) {
    rowmap[id] = -1;
    if (sl == 0) tile_prop[t] = -1;
    return;
  }
  int lo = 0, hi = P - 1;   // smallest p with tile_base[p + 1] > t
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (tile_base[mid + 1] > t) hi = mid;
    else lo = mid + 1;
  }
  const int p = lo;
  const long long i = (long long)(t - tile_base[p]) * tr + sl;
  const long long rows_p = (long long)(sub_base[p + 1] - sub_base[p]) * K;
  rowmap[id] = i < rows_p ? (int)((long long)perm[sub_base[p] + i / K] * K + i % K) : -1;
  if (sl == 0) tile_prop[t] = p;
}

// ------------------------------------------------------------------------------------------
}  // namespace tc

// ------------------------------------------------------------------------------------------
// Host side
// ------------------------------------------------------------------------------------------
using namespace tc;

struct TcNet {
  bool ready = false;
  std::vector<__nv_bfloat16*> bufs;
  Maps maps;
  int box_bwd[MAXL + 1] = {0};
  int box_fwd[MAXL + 1] = {0};
  int woff[MAXL + 1] = {0};
  int mask_words = 0;
  // conv layers on the tensor cores: BF16 weight matrices [Np][Kp] for the backward (rows =
  // input channels) and the forward (rows = output channels), with their TMA maps
  bool conv_ready = false;
};

static std::mutex g_tc_mu;
static std::vector<std::pair<const bcrown_net*, TcNet*>> g_tc;

static TcNet* tc_of(const bcrown_net* net) {
  std::lock_guard<std::mutex> g(g_tc_mu);
  for (auto& e : g_tc)
    if (e.first == net) return e.second;
  TcNet* t = new TcNet();
  g_tc.push_back({net, t});
  return t;
}

bool tc_supported(const bcrown_net* net) {
  if (net->L < 2 || net->L > MAXL) return false;
  if (net->d[0] > MAX_D0) return false;
  int words = 0;
  for (int i = 0; i < net->L; ++i)
    if (net->ly[i].kind != BCROWN_LAYER_FC) return false;
  for (int i = 1; i < net->L; ++i) {
    if (net->d[i] > MAX_HIDDEN) return false;
    words += (net->d[i] + 31) / 32;
  }
  if (words > MAX_MASK_WORDS || net->H > MAX_H) return false;
  // the forward contraction of layer 1 streams d0 in K blocks into accumulators of its own, one per M chunk
  static_assert(MAX_HIDDEN <= NFACC * MCH, "forward layer 1 needs an accumulator per M chunk");
  int dev = 0, major = 0, minor = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return false;
  cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev);
  cudaDeviceGetAttribute(&minor, cudaDevAttrComputeCapabilityMinor, dev);
  cudaGetLastError();
  return major == 10 && minor == 3;
}

static int sm_count() {
  int dev = 0, sms = 148;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return sms;
}

// Tiles the planner can produce: every property may end in one partly filled tile.
static long long max_tiles_of(int B, int K, int P, int tr) { return ((long long)B * K + tr - 1) / tr + P; }

// Rows per tile: the smallest tile whose tiles still get an SM each, since a tile's time is mostly
// its chain of contractions and epilogues (measured on 784-256x6-10, bound and gradient: 59 us at
// 16 rows, 75 at 32, 115 at 64), and 64 where several tiles follow one another on an SM, since a
// row then costs least (9,900 rows of 32 142 us, of 64 119; 19,800 rows 347 / 350).  The results do
// not depend on it: a row is one column of every contraction.
static int tile_rows(int B, int K, int P) {
  const long long sms = sm_count();
  for (int tr : {16, 32})
    if (max_tiles_of(B, K, P, tr) <= sms) return tr;
  return 64;
}

// Workspace: the row plan (counters, prefix sums, permutation, tile -> property, row map), then,
// for the gradient, the BF16 stash [tile][H][TR].
struct TcPlan {
  int *cnt, *cursor, *sub_base, *tile_base, *n_tiles, *perm, *tile_prop, *rowmap;
  __nv_bfloat16* stash;
};
static size_t carve(char* base, int B, int K, int P, int H, bool grad, TcPlan* out) {
  const int tr = tile_rows(B, K, P);
  const long long T = max_tiles_of(B, K, P, tr);
  size_t off = 0;
  auto take = [&](size_t bytes) -> char* {
    char* p = base ? base + off : nullptr;
    off += align_up(bytes);
    return p;
  };
  TcPlan pl;
  pl.cnt = (int*)take((size_t)(P + 1) * 4);
  pl.cursor = (int*)take((size_t)(P + 1) * 4);
  pl.sub_base = (int*)take((size_t)(P + 1) * 4);
  pl.tile_base = (int*)take((size_t)(P + 1) * 4);
  pl.n_tiles = (int*)take(4);
  pl.perm = (int*)take((size_t)std::max(B, 1) * 4);
  pl.tile_prop = (int*)take((size_t)T * 4);
  pl.rowmap = (int*)take((size_t)T * tr * 4);
  pl.stash = grad ? (__nv_bfloat16*)take((size_t)T * tr * std::max(H, 1) * sizeof(__nv_bfloat16)) : nullptr;
  if (out) *out = pl;
  return off;
}

size_t tc_workspace_bytes(const bcrown_net* net, int B, int P, bool grad) {
  return carve(nullptr, B, net->K, P, net->H, grad, nullptr);
}


// BF16 copy of a [rows][cols] FP32 matrix with the row length padded to a multiple of 64.
static int padded_bf16(const float* src_dev, int rows, int cols, __nv_bfloat16** out, int* kp) {
  *kp = (cols + KBLK - 1) / KBLK * KBLK;
  std::vector<float> h((size_t)rows * cols);
  if (cudaMemcpy(h.data(), src_dev, h.size() * 4, cudaMemcpyDeviceToHost) != cudaSuccess)
    return fail(BCROWN_ERR_CUDA, "copy of weights");
  std::vector<__nv_bfloat16> p((size_t)rows * *kp, __float2bfloat16_rn(0.f));
  for (int r = 0; r < rows; ++r)
    for (int c = 0; c < cols; ++c) p[(size_t)r * *kp + c] = __float2bfloat16_rn(h[(size_t)r * cols + c]);
  if (cudaMalloc(out, p.size() * 2) != cudaSuccess) return fail(BCROWN_ERR_OOM, "bf16 weights");
  if (cudaMemcpy(*out, p.data(), p.size() * 2, cudaMemcpyHostToDevice) != cudaSuccess)
    return fail(BCROWN_ERR_CUDA, "bf16 weights upload");
  return BCROWN_OK;
}

template <int MODE, int TR>
static cudaError_t fused_smem() {
  return cudaFuncSetAttribute(k_fused<MODE, TR>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(Smem<TR>) + 1024);
}
template <int MODE>
static void fused_launch(int tr, int grid, const Maps& maps, const Args& A, cudaStream_t s) {
  if (tr == 16) k_fused<MODE, 16><<<grid, NTHREADS, sizeof(Smem<16>) + 1024, s>>>(maps, A);
  else if (tr == 32) k_fused<MODE, 32><<<grid, NTHREADS, sizeof(Smem<32>) + 1024, s>>>(maps, A);
  else k_fused<MODE, 64><<<grid, NTHREADS, sizeof(Smem<64>) + 1024, s>>>(maps, A);
}

static int tc_prepare(bcrown_net* net, TcNet* t) {
  if (t->ready) return BCROWN_OK;
  memset(&t->maps, 0, sizeof(t->maps));
  int w = 0;
  for (int i = 1; i < net->L; ++i) {
    t->woff[i] = w;
    w += (net->d[i] + 31) / 32;
  }
  t->mask_words = w;
  for (int i = 1; i < net->L; ++i) {
    const LayerDev& l = net->ly[i - 1];
    // backward: rows = d_{i-1} output neurons, K = d_i
    __nv_bfloat16* wt = nullptr;
    int kp = 0;
    BC_CHECK(padded_bf16(l.Wt, l.d_in, l.d_out, &wt, &kp));
    t->bufs.push_back(wt);
    t->box_bwd[i] = MCH;
    BC_CHECK(encode_map(&t->maps.bwd[i], wt, l.d_in, kp, t->box_bwd[i]));
    // forward: rows = d_i output neurons, K = d_{i-1}
    __nv_bfloat16* wf = nullptr;
    BC_CHECK(padded_bf16(l.W, l.d_out, l.d_in, &wf, &kp));
    t->bufs.push_back(wf);
    t->box_fwd[i] = MCH;
    BC_CHECK(encode_map(&t->maps.fwd[i], wf, l.d_out, kp, t->box_fwd[i]));
  }
  BC_CUDA((fused_smem<0, 16>()));
  BC_CUDA((fused_smem<0, 32>()));
  BC_CUDA((fused_smem<0, 64>()));
  BC_CUDA((fused_smem<1, 16>()));
  BC_CUDA((fused_smem<1, 32>()));
  BC_CUDA((fused_smem<1, 64>()));
  BC_CUDA((fused_smem<2, 16>()));
  BC_CUDA((fused_smem<2, 32>()));
  BC_CUDA((fused_smem<2, 64>()));
  t->ready = true;
  return BCROWN_OK;
}

static int tc_launch(bcrown_net* net, const bcrown_domain* dom, const bcrown_batch* bt, const Tables& tb, Args& A,
                     char* ws, size_t ws_bytes, int mode, bool plan, cudaStream_t s) {
  const bool grad = mode >= 1;
  TcNet* t = tc_of(net);
  BC_CHECK(tc_prepare(net, t));
  const int B = bt->B, K = net->K, P = dom->n_props;
  const int R = B * K;
  if (R == 0) return BCROWN_OK;
  if (!ws || ws_bytes < tc_workspace_bytes(net, B, P, grad))
    return fail(BCROWN_ERR_OOM, "tensor-core workspace too small");
  TcPlan pl;
  carve(ws, B, K, P, net->H, grad, &pl);
  const int tr = tile_rows(B, K, P);
  const long long T = max_tiles_of(B, K, P, tr);
  // One property: row r is slot r % tr of tile r / tr and no plan is made.  The memset and the four
  // launches of a plan took 13 us of a 77 us call (16 subdomains of the 784-wide network).
  const bool single = P == 1;
  if (plan && !single) {
    BC_CUDA(cudaMemsetAsync(pl.cnt, 0, (size_t)(P + 1) * 4, s));
    const int gb = (int)std::min<long long>((B + 255) / 256, 4096);
    k_plan_count<<<gb, 256, 0, s>>>(B, P, bt->prop_of, pl.cnt, net->status);
    k_plan_scan<<<1, 1024, 0, s>>>(P, K, tr, pl.cnt, pl.cursor, pl.sub_base, pl.tile_base, pl.n_tiles);
    k_plan_scatter<<<gb, 256, 0, s>>>(B, P, bt->prop_of, pl.sub_base, pl.cursor, pl.perm);
    k_plan_rows<<<(int)((T * tr + 255) / 256), 256, 0, s>>>((int)T, K, P, tr, pl.n_tiles, pl.tile_base, pl.sub_base,
                                                           pl.perm, pl.tile_prop, pl.rowmap);
    g_launches += 4;
  }
  A.L = net->L;
  A.K = K;
  A.P = P;
  A.H = net->H;
  A.R = R;
  A.tiles = (int)(((long long)R + tr - 1) / tr);
  A.n_tiles = single ? nullptr : pl.n_tiles;
  A.tile_prop = pl.tile_prop;
  A.rowmap = pl.rowmap;
  A.stash = pl.stash;
  for (int i = 0; i <= net->L && i <= MAXL; ++i) A.d[i] = net->d[i];
  for (int i = 1; i < net->L; ++i) {
    A.hoff[i] = net->hoff[i - 1];
    A.woff[i] = t->woff[i];
    A.bias[i] = net->ly[i - 1].b;
    A.box_bwd[i] = t->box_bwd[i];
    A.box_fwd[i] = t->box_fwd[i];
  }
  A.mask_words = t->mask_words;
  A.Wbar = net->Wbar;
  A.bbar = net->bbar;
  A.bt = BatchView{bt->B, bt->prop_of, bt->split_off, bt->split_cnt, bt->split_layer, bt->split_idx, bt->split_sign,
                   bt->alpha_off};
  A.tb = tb;
  A.x_lo = dom->x_lo;
  A.x_hi = dom->x_hi;
  A.n_alpha = bt->n_alpha;
  A.n_beta = bt->n_beta;
  A.status = net->status;
  // one CTA per SM at most; the planned tile count (at most T) is read on the device
  const int grid = (int)std::min<long long>(single ? A.tiles : T, sm_count());
  {
    ProfScope ps(net, BCROWN_PROF_FUSED, s);
    if (mode == 2) fused_launch<2>(tr, grid, t->maps, A, s);
    else if (mode == 1) fused_launch<1>(tr, grid, t->maps, A, s);
    else fused_launch<0>(tr, grid, t->maps, A, s);
    ++g_launches;
  }
  BC_CUDA(cudaGetLastError());
  return BCROWN_OK;
}

int tc_bound(bcrown_net* net, const bcrown_domain* dom, const bcrown_batch* bt, const Tables& tb, char* ws,
             size_t ws_bytes, bool grad, bool plan, const float* alpha, const float* beta, float* lb, float* dalpha,
             float* dbeta, cudaStream_t s, __nv_bfloat16* dalpha16) {
  Args A;
  memset(&A, 0, sizeof(A));
  A.alpha = alpha;
  A.beta = beta;
  A.lb = lb;
  A.dalpha = dalpha;
  A.dalpha16 = dalpha16;
  A.dbeta = dbeta;
  return tc_launch(net, dom, bt, tb, A, ws, ws_bytes, !grad ? 0 : (dalpha16 ? 2 : 1), plan, s);
}

void tc_release(const bcrown_net* net) {
  std::lock_guard<std::mutex> g(g_tc_mu);
  for (size_t i = 0; i < g_tc.size(); ++i)
    if (g_tc[i].first == net) {
      for (auto* b : g_tc[i].second->bufs) cudaFree(b);
      delete g_tc[i].second;
      g_tc.erase(g_tc.begin() + i);
      return;
    }
}

}  // namespace bcrown
