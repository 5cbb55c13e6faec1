// The FP32 bound and gradient of a small fully connected network in one launch: a row (subdomain,
// specification) walks its whole chain -- the tables of its property, relaxation and contraction of
// every layer, concretisation, the minimising corner and the adjoint pass -- with everything but the
// weights in shared memory.
//
// Layer by layer the path is a launch or two per layer and pass, each of a few blocks: 16-32-32-4,
// 192 rows, bound and gradient: 12 launches, 57 us, of which no kernel has 2 us of work.  Here a
// warp takes the row (four rows a block) where no layer is wider than ROWS_WARP_WIDTH, else a block
// of 256 threads; a thread owns every 32nd or 256th output of a contraction.  Bound by the latency of the
// weights' loads, so 16 of them are in flight per thread (8 where the rows fill the chip).
//
// Every sum has the order that the layers' kernels give it (the GEMM's chain over k, the relaxation's
// lanes, the concretisation's 256 threads), so a row's bits do not depend on the kernel, and with it
// on the batch.
#include <algorithm>
#include <atomic>

#include "simt.cuh"

namespace bcrown {

extern std::atomic<long long> g_launches;

namespace {

constexpr int ROWS_MAXL = 16;          // layers
constexpr int ROWS_H = 2048;           // hidden neurons
constexpr int ROWS_D0 = 2048;          // inputs
constexpr int ROWS_WIDTH = 512;        // widest hidden layer
constexpr int ROWS_WARP_WIDTH = 64;    // widest layer of the form with one warp per row
constexpr int ROWS_BLOCK = 256, ROWS_WARP_ROWS = 4;

struct RowsNet {
  int L, H, mw;                        // mw: widest layer, the input included
  int d[ROWS_MAXL + 1], hoff[ROWS_MAXL + 1];
  const float *W[ROWS_MAXL + 1], *Wt[ROWS_MAXL + 1], *b[ROWS_MAXL + 1];
  const float *Wbar, *bbar;
};

// H and mw rounded up to a multiple of 4, so that Lam, h and z lie on 16-byte boundaries
__host__ __device__ constexpr int rows_pad(int x) { return (x + 3) & ~3; }
__host__ __device__ constexpr int rows_floats(int H, int mw) { return 5 * rows_pad(H) + 3 * rows_pad(mw); }

template <int T>
__device__ __forceinline__ void row_sync() {
  if (T > 32) __syncthreads();
  else __syncwarp();
}

// y[n] = sum_k x[k] w[k][n] over n = t, t + T, ..: store(n, sum).  One chain over k whatever V, the loads
// of V terms in flight (x 16-byte aligned, read 4 terms at a time).
template <int T, int V, class F>
__device__ __forceinline__ void row_product(const float* x, const float* __restrict__ w, int K, int N, int t, F store) {
#pragma unroll 1
  for (int n = t; n < N; n += T) {
    const float* wp = w + n;
    float acc = 0.f;
    int k = 0;
#pragma unroll 1
    for (; k + V <= K; k += V, wp += (size_t)V * N) {
      float wv[V];
      float4 xv[V / 4];
#pragma unroll
      for (int e = 0; e < V; ++e) wv[e] = __ldg(wp + (size_t)e * N);
#pragma unroll
      for (int e = 0; e < V / 4; ++e) xv[e] = *reinterpret_cast<const float4*>(x + k + 4 * e);
#pragma unroll
      for (int e = 0; e < V / 4; ++e) {
        acc = fmaf(xv[e].x, wv[4 * e], acc);
        acc = fmaf(xv[e].y, wv[4 * e + 1], acc);
        acc = fmaf(xv[e].z, wv[4 * e + 2], acc);
        acc = fmaf(xv[e].w, wv[4 * e + 3], acc);
      }
    }
    if (k < K) {   // the rest, its loads together as well
      float wv[V];
#pragma unroll
      for (int e = 0; e < V; ++e) wv[e] = k + e < K ? __ldg(wp + (size_t)e * N) : 0.f;
#pragma unroll
      for (int e = 0; e < V; ++e)
        if (k + e < K) acc = fmaf(x[k + e], wv[e], acc);
    }
    store(n, acc);
  }
}

// sum_j Lam[j] b[j] + a[j] lm[j] over the lanes of a warp, in the order of the layers' relaxation pass: 4
// neighbours at a time per lane where d is a multiple of 4, else every 32nd, then the same exchange.
// All operands lie in shared memory.
__device__ __forceinline__ float row_bias_sum(const float* Lam, const float* b, const float* a, const float* lm, int d,
                                              int lane) {
  float acc = 0.f;
  if ((d & 3) == 0) {
    for (int j = 4 * lane; j < d; j += 128)
#pragma unroll
      for (int v = 0; v < 4; ++v) acc = fmaf(Lam[j + v], b[j + v], fmaf(a[j + v], lm[j + v], acc));
  } else {
    for (int j = lane; j < d; j += 32) acc = fmaf(Lam[j], b[j], fmaf(a[j], lm[j], acc));
  }
  return warp_sum(acc);
}

// T: threads per row, 32 (ROWS_WARP_ROWS rows a block) or the block.  V: weights in flight a thread; the
// block form with 16 asks for 3 blocks an SM only (62 registers, 4 fit): without that the compiler keeps to
// the registers of more blocks and issues fewer of the loads together.
template <int T, int V>
__global__ void __launch_bounds__(T == 32 ? 32 * ROWS_WARP_ROWS : T, T > 32 && V == 16 ? 3 : 0)
    k_rows(const RowsNet net, RowsCtx c, const float* __restrict__ alpha, int64_t n_alpha,
           const float* __restrict__ beta, int64_t n_beta, float* __restrict__ lb, float* __restrict__ xstar,
           bool grad, float* __restrict__ dalpha, float* __restrict__ dbeta) {
  extern __shared__ __align__(16) float rows_smem[];
  __shared__ float red[T > 32 ? 32 : 1];
  __shared__ float part[T > 32 ? ROWS_MAXL + 1 : 1];   // the layers' bias sums
  __shared__ int tot[T / 32];
  const int t = threadIdx.x % T, lane = threadIdx.x & 31, w = t >> 5;
  const int rl = blockIdx.x * (T == 32 ? ROWS_WARP_ROWS : 1) + threadIdx.x / T;
  if (rl >= c.R) return;   // (whole rows: a warp, or no thread of the block)
  const int H = net.H, L = net.L;
  float* A = rows_smem + (size_t)(threadIdx.x / T) * rows_floats(H, net.mw);
  const int Hp = rows_pad(H), mwp = rows_pad(net.mw);
  float *D = A + Hp, *lm = D + Hp;
  int *rank = reinterpret_cast<int*>(lm + Hp), *sp = rank + Hp;
  float *Lam = reinterpret_cast<float*>(sp + Hp), *h = Lam + mwp, *z = h + mwp;

  int b, k, p;
  const bool ok = row_prop(c, rl, &b, &k, &p);
  if (!ok) {
    if (t == 0) flag(c.status, BCROWN_ERR_ARG);
    p = 0;
  }
  const int off = c.bt.split_off[b], cnt = c.bt.split_cnt[b];
  if ((cnt < 0 || cnt > BCROWN_MAX_SPLITS) && t == 0) flag(c.status, BCROWN_ERR_ARG);
  const int ns = cnt < 0 || cnt > BCROWN_MAX_SPLITS ? 0 : cnt;

  // the property's table (as k_tables): D, lambda of a stable neuron, the chord and the rank of an unstable one
  const float *lp = c.l + (size_t)p * H, *up = c.u + (size_t)p * H;
  int U = 0;
  for (int n0 = 0; n0 < H; n0 += T) {
    const int n = n0 + t;
    const float lv = n < H ? lp[n] : 0.f, uv = n < H ? up[n] : 0.f;
    const bool un = n < H && is_unstable(lv, uv);
    const unsigned m = __ballot_sync(0xffffffffu, un);
    int r = U + __popc(m & ((1u << lane) - 1u));
    U += __popc(m);
    if (T > 32) {
      U -= __popc(m);
      if (lane == 0) tot[w] = __popc(m);
      __syncthreads();
      int all = 0;
#pragma unroll
      for (int q = 0; q < T / 32; ++q) {
        if (q < w) r += tot[q];
        all += tot[q];
      }
      U += all;
      __syncthreads();
    }
    if (n < H) {
      const float sl = un ? __fdiv_ru(uv, __fsub_rd(uv, lv)) : (lv >= 0.f ? 1.f : 0.f);
      rank[n] = un ? r : -1;
      D[n] = sl;
      lm[n] = un ? __fmul_ru(sl, -lv) : 0.f;
      sp[n] = 0;
    }
  }
  for (int j = t; j < net.d[L - 1]; j += T) (L > 1 ? A + net.hoff[L - 1] : h)[j] = net.Wbar[(size_t)k * net.d[L - 1] + j];
  row_sync<T>();
  // the row's splits: sp = 2 (place in the list + 1) + (sign > 0), the last of a neuron's
  for (int q = t; q < ns; q += T) {
    const int ly = c.bt.split_layer[off + q], sg = c.bt.split_sign[off + q];
    const long long j = c.bt.split_idx[off + q];
    if (sg != -1 && sg != 1) flag(c.status, BCROWN_ERR_ARG);
    else if (ly >= 1 && ly < L) {
      if (j >= net.d[ly]) flag(c.status, BCROWN_ERR_ARG);
      else atomicMax(sp + net.hoff[ly] + (int)j, 2 * (q + 1) + (sg > 0 ? 1 : 0));
    }
  }
  row_sync<T>();

  const long long abase = c.bt.alpha_off[b] + (long long)k * U;
  const long long bbase = (long long)off * c.K + (long long)k * cnt;
  float c0 = ok ? net.bbar[k] : -INFINITY;
  for (int i = L - 1; i >= 1; --i) {
    const int d = net.d[i], o = net.hoff[i];
    for (int j = t; j < d; j += T) {
      const int n = o + j, s2 = sp[n];
      const float a = A[n];
      z[j] = net.b[i][j];   // (z is free until the adjoint pass)
      float Dn = D[n], ln = lm[n], bs = 0.f;
      if (s2) {
        const long long bi = bbase + (s2 >> 1) - 1;
        const float sg = s2 & 1 ? 1.f : -1.f;
        if (bi >= 0 && bi < n_beta) bs = fmaxf(beta[bi], 0.f) * sg;
        else flag(c.status, BCROWN_ERR_ARG);
        Dn = s2 & 1 ? 0.f : 1.f;
        ln = 0.f;
      } else if (rank[n] >= 0 && a >= 0.f) {
        const long long ai = abase + rank[n];
        ln = 0.f;
        if (ai < 0 || ai >= n_alpha) {
          flag(c.status, BCROWN_ERR_ARG);
          Dn = 0.f;
        } else {
          Dn = fminf(fmaxf(alpha[ai], 0.f), 1.f);
        }
      }
      D[n] = Dn;
      lm[n] = ln;
      Lam[j] = fmaf(a, Dn, bs);
    }
    row_sync<T>();
    if (T == 32) {
      c0 += row_bias_sum(Lam, z, A + o, lm + o, d, lane);
    } else if (w == i % (T / 32)) {   // one warp of the block, another each layer
      const float sum = row_bias_sum(Lam, z, A + o, lm + o, d, lane);
      if (lane == 0) part[i] = sum;
    }
    float* out = i > 1 ? A + net.hoff[i - 1] : h;
    row_product<T, V>(Lam, net.W[i], d, net.d[i - 1], t, [&](int n, float v) { out[n] = v + 0.f; });   // (-0 as the GEMM's 0)
    row_sync<T>();
  }
  // concretisation, and the corner that attains it
  const float *xl = c.x_lo + (size_t)p * net.d[0], *xh = c.x_hi + (size_t)p * net.d[0];
  // (summed as by 256 threads: in the warp's form, whose inputs are at most 64, by two warps of them)
  float s0 = 0.f, s1 = 0.f;
  for (int m = t; m < net.d[0]; m += T) {
    const float a = h[m], v = fminf(a * xl[m], a * xh[m]);
    if (T > 32 || m < 32) s0 += v;
    else s1 += v;
    const float x = a >= 0.f ? xl[m] : xh[m];
    if (xstar) xstar[(size_t)(c.r0 + rl) * net.d[0] + m] = x;
    h[m] = x;
  }
  if (T > 32) {
    s0 = block_sum(s0, red);
    for (int i = L - 1; i >= 1; --i) c0 += part[i];
  } else {
    s0 = (warp_sum(s0) + 0.f) + (warp_sum(s1) + 0.f);
    __syncwarp();
  }
  if (t == 0) {
    float out = c0 + s0;
    if (!isfinite(out)) {
      flag(c.status, BCROWN_ERR_NONFINITE);
      out = -INFINITY;
    }
    lb[c.r0 + rl] = out;
  }
  if (!grad) return;
  for (int i = 1; i < L; ++i) {
    const int o = net.hoff[i];
    row_product<T, V>(h, net.Wt[i], net.d[i - 1], net.d[i], t, [&](int j, float v) {
      const int n = o + j, s2 = sp[n];
      const float zj = v + net.b[i][j], a = A[n];
      if (rank[n] >= 0) {
        const long long ai = abase + rank[n];
        if (ai < 0 || ai >= n_alpha) flag(c.status, BCROWN_ERR_ARG);
        else dalpha[ai] = !s2 && a >= 0.f ? a * zj : 0.f;
      }
      if (s2) {
        const long long bi = bbase + (s2 >> 1) - 1;
        if (bi >= 0 && bi < n_beta) dbeta[bi] = s2 & 1 ? zj : -zj;
        else flag(c.status, BCROWN_ERR_ARG);
      }
      z[j] = fmaf(D[n], zj, lm[n]);
    });
    row_sync<T>();
    float* sw = h;
    h = z;
    z = sw;
  }
}

int widest(const bcrown_net* net) {
  int w = net->d[0];
  for (int i = 1; i < net->L; ++i) w = std::max(w, net->d[i]);
  return w;
}

}  // namespace

int rows_load(const bcrown_net* net) {
  if (!rows_supported(net, 0, false) && !rows_supported(net, 0, true)) return BCROWN_OK;
  const int smem = rows_floats(ROWS_H, ROWS_D0) * 4;
  for (cudaError_t e : {cudaFuncSetAttribute(k_rows<ROWS_BLOCK, 8>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem),
                        cudaFuncSetAttribute(k_rows<ROWS_BLOCK, 16>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem),
                        cudaFuncSetAttribute(k_rows<32, 16>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem)})
    if (e != cudaSuccess) return fail(BCROWN_ERR_CUDA, "row kernel: shared memory");
  return BCROWN_OK;
}

// Rows of the block form that are resident at once with 16 loads in flight (4 blocks on each of 152 SMs);
// more go 8 at a time, in more blocks.
constexpr int ROWS_DEEP = 608;

// Which calls take it.  A row's bits are the same either way: the sums have the layers' order.
// Times of calls, bound / bound and gradient, here and layer by layer (us; below 26 the host's time):
//   16-32-32-4       192 rows 23 / 29, 40 / 57;  8,192 22 / 30, 59 / 102;  196,608 217 / 293, 618 / 1,337
//   64x4-10          2,048 rows 24 / 35, 55 / 104;  196,608 698 / 1,249, 1,023 / 2,445
//   64x9-10          8,192 rows 134 / 238, 157 / 344;  32,768 506 / 929, 396 / 958
//   37-300-260-5     64 rows 24 / 36, 63 / 102;  1,024 40 / 76, 67 / 106;  1,400 64 / 117, 69 / 113
//   784-256x6-10     8 rows 51 / 88, 125 / 246;  72 53 / 90, 120 / 240
//   784-20-10        2,048 rows 23 / 61, 39 / 80;  8,192 67 / 195, 59 / 131
//   2048-16-10       1,024 rows 24 / 67, 37 / 117;  2,048 31 / 130, 38 / 129
//   2048-20-512-3    1,024 rows 61 / 162, 63 / 160;  2,048 91 / 244, 71 / 178
//   1024-512-10      8 rows 41 / 75, 42 / 88;  2048-512-4  8 rows 73 / 138, 44 / 118
// The warp form gains everywhere but where many hidden neurons leave few rows resident (64x9: 11 KB a
// row), from 2^28 FMAs a pass on.  The block form reads the weights once per row: it is for the rows that
// leave the GEMM's tiles empty, by their FMAs a pass (a layer's launches buy 2^26 of them) and the terms
// of their chains; and for layers whose own chains (one after the other over the outputs that a thread
// owns) are not longer than a layer's launches take, the bound's and the gradient's apart.
constexpr long long ROWS_FMAS = 1LL << 27, ROWS_LAYER_FMAS = 1LL << 26, ROWS_WARP_FMAS = 1LL << 28;
constexpr long long ROWS_TERMS = 3LL << 20;
constexpr int ROWS_BOUND_TERMS = 1536, ROWS_GRAD_TERMS = 4096;

static bool warp_form(const bcrown_net* net) { return widest(net) <= ROWS_WARP_WIDTH && net->H <= ROWS_H / 4; }

bool rows_supported(const bcrown_net* net, long long R, bool grad) {
  if (net->L > ROWS_MAXL || net->H > ROWS_H || net->d[0] > ROWS_D0) return false;
  long long fma = 0, back = 0, fwd = 0;   // FMAs of a pass; terms in a row's chains, one after the other
  for (int i = 1; i < net->L; ++i) {
    const int in = net->d[i - 1], out = net->d[i];
    if (net->ly[i - 1].kind != BCROWN_LAYER_FC || out > ROWS_WIDTH) return false;
    fma += (long long)out * in;
    back += (long long)((in + ROWS_BLOCK - 1) / ROWS_BLOCK) * out;
    fwd += (long long)((out + ROWS_BLOCK - 1) / ROWS_BLOCK) * in;
  }
  const int n = net->L - 1;
  if (warp_form(net)) return widest(net) <= 32 || net->H <= 256 || R * fma <= ROWS_WARP_FMAS;
  return R * fma <= std::min(n * ROWS_LAYER_FMAS, ROWS_FMAS) && R * (back + fwd) <= ROWS_TERMS &&
         (grad ? back + fwd <= (long long)n * ROWS_GRAD_TERMS : back <= (long long)n * ROWS_BOUND_TERMS);
}

int rows_bound(const bcrown_net* net, const RowsCtx& c, const float* alpha, int64_t n_alpha, const float* beta,
               int64_t n_beta, float* lb, float* xstar, bool grad, float* dalpha, float* dbeta, cudaStream_t s) {
  RowsNet n{};
  n.L = net->L;
  n.H = net->H;
  n.mw = widest(net);
  n.Wbar = net->Wbar;
  n.bbar = net->bbar;
  for (int i = 0; i < net->L; ++i) n.d[i] = net->d[i];
  for (int i = 1; i < net->L; ++i) {
    n.hoff[i] = (int)net->hoff[i - 1];
    n.W[i] = net->ly[i - 1].W;
    n.Wt[i] = net->ly[i - 1].Wt;
    n.b[i] = net->ly[i - 1].b;
  }
  const int smem = rows_floats(n.H, n.mw) * 4;
  auto go = [&](auto* kernel, int rows, int threads) {
    kernel<<<(c.R + rows - 1) / rows, threads, rows * smem, s>>>(n, c, alpha, n_alpha, beta, n_beta, lb, xstar, grad,
                                                                 dalpha, dbeta);
  };
  if (warp_form(net)) go(k_rows<32, 16>, ROWS_WARP_ROWS, 32 * ROWS_WARP_ROWS);
  else if (c.R <= ROWS_DEEP) go(k_rows<ROWS_BLOCK, 16>, 1, ROWS_BLOCK);
  else go(k_rows<ROWS_BLOCK, 8>, 1, ROWS_BLOCK);
  ++g_launches;
  return BCROWN_OK;
}

}  // namespace bcrown
