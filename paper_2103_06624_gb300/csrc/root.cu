// Root intermediate bounds (Section 3.3; CROWN, Lemma 2.2, beta' = 0): rows (property, +-, j) of one
// hidden layer T, back-substituted through layers T-1 .. 1 and concretised.
//
// - Layer 1 is the exact interval of an affine map: one warp per neuron sums min(w x_lo, w x_hi)
//   over the neuron's own weights.
// - Layer T >= 2 starts from A^(T-1) = +-(row j of W^(T)), copied: no contraction of unit vectors.
// - Where layers 1 .. T are convolutions, row j of layer T reaches only its receptive field: A^(m)
//   is kept as the patch [C_m][n_m][n_m] around it (n_T = 1, n_(m-1) = (n_m - 1) s_m + k_m), and
//   each contraction is the transposed convolution of the patch (no padding).  Positions of the
//   patch outside the map are no neurons: their A is dropped at the next relaxation.
// - The rows of all properties run together.
//
// Bound by HBM (the A rows of the SIMT path) and by the FP32 contractions.  On the 3x32x32 ->
// conv32 -> conv64 -> 512-512-10 network (4x4 stride 2), contracting unit vectors through dense maps
// took 1.8 ms for layer 1 (now 10 us) and 2.5 ms for layer 2, whose rows hold 512 of 8192 and
// 300 of 3072 values.
#include <algorithm>
#include <atomic>

#include "simt.cuh"

namespace bcrown {

extern std::atomic<long long> g_launches;

// Row rl of the chunk: property, +1 / -1, target neuron.
struct RootRow {
  int p, j;
  float sg;
};
__device__ __forceinline__ RootRow root_row(const RootCtx& c, int rl) {
  const long long g = c.g0 + rl;
  RootRow r;
  r.p = (int)(g / (2 * c.d_top));
  const int q = (int)(g - (long long)r.p * 2 * c.d_top);
  r.j = q < c.d_top ? q : q - c.d_top;
  r.sg = q < c.d_top ? 1.f : -1.f;
  return r;
}

__device__ __forceinline__ void root_write(const RootCtx& c, const RootRow& r, float out) {
  const size_t n = (size_t)r.p * c.H + c.hoff_top + r.j;
  if (r.sg > 0.f) c.l[n] = isfinite(out) ? out : -INFINITY;
  else c.u[n] = isfinite(out) ? -out : INFINITY;
}

// Layer 1: one warp per (property, neuron), both directions.
template <bool CERT>
__global__ void __launch_bounds__(256) k_root_first(RootCtx c, LayerGeom g, const float* __restrict__ W,
                                                    const float* __restrict__ b, long long total) {
  const long long id = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (id >= total) return;
  const int p = (int)(id / g.d_out), j = (int)(id - (long long)p * g.d_out);
  const float* xl = c.x_lo + (size_t)p * c.d0;
  const float* xh = c.x_hi + (size_t)p * c.d0;
  float s0 = 0.f, s1 = 0.f;   // sums for +z_j and -z_j
  auto term = [&](float w, int m) {
    const float lo = xl[m], hi = xh[m];
    if (CERT) {
      // products rounded down, then summed rounded down: a lower bound of sum_m min(...)
      s0 = __fadd_rd(s0, fminf(__fmul_rd(w, lo), __fmul_rd(w, hi)));
      s1 = __fadd_rd(s1, fminf(__fmul_rd(-w, lo), __fmul_rd(-w, hi)));
    } else {
      s0 += fminf(w * lo, w * hi);
      s1 += fminf(-w * lo, -w * hi);
    }
  };
  if (g.kind == BCROWN_LAYER_FC) {
    const float* w = W + (size_t)j * g.d_in;
#pragma unroll 4
    for (int m = lane; m < g.d_in; m += 32) term(w[m], m);
  } else {
    const int hw = g.out_h * g.out_w;
    const int co = j / hw, rem = j - co * hw, oy = rem / g.out_w, ox = rem - oy * g.out_w;
    const int kk = g.k * g.k;
    for (int t = lane; t < g.in_c * kk; t += 32) {
      const int ci = t / kk, r = t - ci * kk, ky = r / g.k, kx = r - ky * g.k;
      const int iy = oy * g.stride - g.pad + ky, ix = ox * g.stride - g.pad + kx;
      if (iy < 0 || iy >= g.in_h || ix < 0 || ix >= g.in_w) continue;
      term(W[(size_t)co * g.in_c * kk + t], (ci * g.in_h + iy) * g.in_w + ix);
    }
  }
  for (int o = 16; o > 0; o >>= 1) {
    s0 = CERT ? __fadd_rd(s0, __shfl_xor_sync(0xffffffffu, s0, o)) : s0 + __shfl_xor_sync(0xffffffffu, s0, o);
    s1 = CERT ? __fadd_rd(s1, __shfl_xor_sync(0xffffffffu, s1, o)) : s1 + __shfl_xor_sync(0xffffffffu, s1, o);
  }
  if (lane != 0) return;
  const float bj = b[j];
  const float o0 = CERT ? __double2float_rd(__dadd_rd((double)bj, (double)s0)) : bj + s0;
  const float o1 = CERT ? __double2float_rd(__dadd_rd((double)-bj, (double)s1)) : -bj + s1;
  root_write(c, RootRow{p, j, 1.f}, o0);
  root_write(c, RootRow{p, j, -1.f}, o1);
}

// A^(T-1) = +-(row j of W^(T)): dense, or with `patch` the k x k patch of every input channel.
__global__ void __launch_bounds__(128) k_root_top(RootCtx c, LayerGeom g, int patch, const float* __restrict__ W,
                                                  const float* __restrict__ b, float* __restrict__ A,
                                                  float* __restrict__ cf, double* __restrict__ cd,
                                                  double* __restrict__ E) {
  const int rl = blockIdx.x;
  const RootRow r = root_row(c, rl);
  const int kk = g.k * g.k;
  if (g.kind == BCROWN_LAYER_FC || patch) {
    const int d = patch ? g.in_c * kk : g.d_in;
    const float* w = W + (size_t)(patch ? r.j / (g.out_h * g.out_w) : r.j) * d;
    for (int m = threadIdx.x; m < d; m += blockDim.x) A[(size_t)rl * d + m] = r.sg * w[m];
  } else {
    const int hw = g.out_h * g.out_w, ihw = g.in_h * g.in_w;
    const int co = r.j / hw, rem = r.j - co * hw, oy = rem / g.out_w, ox = rem - oy * g.out_w;
    for (int m = threadIdx.x; m < g.d_in; m += blockDim.x) {
      const int ci = m / ihw, pos = m - ci * ihw, y = pos / g.in_w, x = pos - y * g.in_w;
      const int ky = y - (oy * g.stride - g.pad), kx = x - (ox * g.stride - g.pad);
      const bool in = ky >= 0 && ky < g.k && kx >= 0 && kx < g.k;
      A[(size_t)rl * g.d_in + m] = in ? r.sg * W[((size_t)co * g.in_c + ci) * kk + ky * g.k + kx] : 0.f;
    }
  }
  if (threadIdx.x == 0) {
    const float bv = r.sg * b[r.j];
    cf[rl] = bv;
    cd[rl] = (double)bv;
    E[rl] = 0.0;
  }
}

// Element e of a row: its neuron (or input) index, -1 outside the map.
__device__ __forceinline__ int root_index(const RootMap& m, int oy, int ox, int e) {
  if (!m.n) return e;
  const int ch = (int)m.dnn((uint32_t)e), rem = e - ch * m.n * m.n, ey = (int)m.dn((uint32_t)rem), ex = rem - ey * m.n;
  const int y = oy + ey, x = ox + ex;
  return (unsigned)y < (unsigned)m.Hm && (unsigned)x < (unsigned)m.Wm ? (ch * m.Hm + y) * m.Wm + x : -1;
}
// Origin of the row's patch in map m: an affine function of the target neuron's position.
__device__ __forceinline__ void root_origin(const RootCtx& c, const RootMap& m, int j, int* oy, int* ox) {
  *oy = *ox = 0;
  if (!m.n) return;
  const int pos = j % (c.top_h * c.top_w);
  *oy = (pos / c.top_w) * m.os - m.oo;
  *ox = (pos % c.top_w) * m.os - m.oo;
}

// Relaxation of hidden layer m for root rows (no splits, alpha' from the rule), one block per row.
// The chord is worked out from l, u here with the tables' outward rounding: the loads are needed
// for the error terms anyway, and the layers' tables need not be rebuilt for every T.
//
// Bound by the latency of its loads (A, l, u, bias and the error weight per element).  A thread takes
// four elements at a time with all their loads issued together: four neighbours by 16-byte loads
// where the row is the whole map and every array lies on a 16-byte boundary (VEC), else four a block
// apart.  1,024 rows of 8,192 neurons, certified: 62 us one element at a time, 28 now; 8,192 patches
// of 512 elements 44, 46 now.
template <bool CERT, bool VEC>
__global__ void __launch_bounds__(256) k_root_relax(RootCtx c, RootMap m, int d, long long hoff, int rule,
                                                    float rule_value, const float* __restrict__ Ain,
                                                    float* __restrict__ Lam, const float* __restrict__ bias,
                                                    float* __restrict__ cf, double* __restrict__ cd,
                                                    double* __restrict__ E, const float* __restrict__ wm,
                                                    double gamma) {
  __shared__ float shf[3][8];
  const int rl = blockIdx.x;
  const RootRow r = root_row(c, rl);
  int oy, ox;
  root_origin(c, m, r.j, &oy, &ox);
  const float* a_row = Ain + (size_t)rl * d;
  float* lam_row = Lam + (size_t)rl * d;
  const size_t n0 = (size_t)r.p * c.H + hoff;
  const float *lp = c.l + n0, *up = c.u + n0, *wp = wm + n0;
  const int nt = blockDim.x;
  // CERT: acc rounded down, e1 and e2 rounded up (as in k_relax)
  float acc = 0.f, e1 = 0.f, e2 = 0.f;
  auto four = [&](const float (&a)[4], const float (&lv)[4], const float (&uv)[4], const float (&bj)[4],
                  const float (&wj)[4], const bool (&in)[4], float (&L)[4]) {
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      L[v] = 0.f;
      if (!in[v]) continue;
      const bool unst = lv[v] < 0.f && uv[v] > 0.f;
      float D = lv[v] >= 0.f ? 1.f : 0.f, lm = 0.f;
      if (unst) {
        if (a[v] >= 0.f) {
          D = rule == BCROWN_ALPHA_ADAPTIVE ? (uv[v] >= -lv[v] ? 1.f : 0.f) : rule_value;
        } else {
          D = __fdiv_ru(uv[v], __fsub_rd(uv[v], lv[v]));
          lm = __fmul_ru(D, -lv[v]);
        }
      }
      L[v] = a[v] * D;
      if (CERT) {
        acc = __fadd_rd(acc, __fadd_rd(__fmul_rd(L[v], bj[v]), __fmul_rd(a[v], lm)));
        if (!(D == 0.f || D == 1.f)) {
          const float zmax = fmaxf(fabsf(lv[v]), fabsf(uv[v]));
          const float er = __fmaf_ru(fabsf(L[v]), 0x1p-23f, 0x1p-140f);
          e1 = __fadd_ru(e1, __fmul_ru(er, zmax));
        }
        e2 = __fadd_ru(e2, __fmul_ru(fabsf(L[v]), wj[v]));
      } else {
        acc = fmaf(L[v], bj[v], fmaf(a[v], lm, acc));
      }
    }
  };
  float a[4], lv[4], uv[4], bj[4], wj[4], L[4];
  bool in[4];
  if (VEC) {
    auto ld4 = [](const float* q, float (&o)[4]) {
      const float4 x = *reinterpret_cast<const float4*>(q);
      o[0] = x.x, o[1] = x.y, o[2] = x.z, o[3] = x.w;
    };
#pragma unroll 2
    for (int e = 4 * threadIdx.x; e < d; e += 4 * nt) {
      ld4(a_row + e, a);
      ld4(lp + e, lv);
      ld4(up + e, uv);
      ld4(bias + e, bj);
      if (CERT) ld4(wp + e, wj);
      in[0] = in[1] = in[2] = in[3] = true;
      four(a, lv, uv, bj, wj, in, L);
      *reinterpret_cast<float4*>(lam_row + e) = make_float4(L[0], L[1], L[2], L[3]);
    }
  } else {
    for (int e0 = threadIdx.x; e0 < d; e0 += 4 * nt) {
#pragma unroll
      for (int v = 0; v < 4; ++v) {
        const int e = e0 + v * nt;
        const int j = e < d ? root_index(m, oy, ox, e) : -1;
        in[v] = j >= 0;
        const int jj = in[v] ? j : 0;
        a[v] = in[v] ? a_row[e] : 0.f;
        lv[v] = lp[jj];
        uv[v] = up[jj];
        bj[v] = bias[jj];
        wj[v] = CERT ? wp[jj] : 0.f;
      }
      four(a, lv, uv, bj, wj, in, L);
#pragma unroll
      for (int v = 0; v < 4; ++v)
        if (e0 + v * nt < d) lam_row[e0 + v * nt] = L[v];
    }
  }
  for (int o = 16; o > 0; o >>= 1) {
    acc = CERT ? __fadd_rd(acc, __shfl_xor_sync(0xffffffffu, acc, o)) : acc + __shfl_xor_sync(0xffffffffu, acc, o);
    if (CERT) {
      e1 = __fadd_ru(e1, __shfl_xor_sync(0xffffffffu, e1, o));
      e2 = __fadd_ru(e2, __shfl_xor_sync(0xffffffffu, e2, o));
    }
  }
  const int w = threadIdx.x >> 5;
  if ((threadIdx.x & 31) == 0) {
    shf[0][w] = acc;
    shf[1][w] = e1;
    shf[2][w] = e2;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int q = 1; q < (nt + 31) / 32; ++q) {
      acc = CERT ? __fadd_rd(acc, shf[0][q]) : acc + shf[0][q];
      e1 = __fadd_ru(e1, shf[1][q]);
      e2 = __fadd_ru(e2, shf[2][q]);
    }
    if (CERT) {
      cd[rl] = __dadd_rd(cd[rl], (double)acc);
      E[rl] = __dadd_ru(E[rl], __dadd_ru((double)e1, __dmul_ru(gamma, (double)e2)));
    } else {
      cf[rl] += acc;
    }
  }
}

template <bool CERT>
__global__ void __launch_bounds__(256) k_root_concretize(RootCtx c, RootMap m, int d, const float* __restrict__ A0,
                                                         const float* __restrict__ cf, const double* __restrict__ cd,
                                                         const double* __restrict__ E) {
  __shared__ float shf[32];
  const int rl = blockIdx.x;
  const RootRow r = root_row(c, rl);
  int oy, ox;
  root_origin(c, m, r.j, &oy, &ox);
  const float* a = A0 + (size_t)rl * d;
  const float* xl = c.x_lo + (size_t)r.p * c.d0;
  const float* xh = c.x_hi + (size_t)r.p * c.d0;
  float s = 0.f;
  for (int e0 = threadIdx.x; e0 < d; e0 += 4 * blockDim.x) {   // four elements' loads in flight
    float am[4], lo[4], hi[4];
    bool in[4];
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      const int e = e0 + v * blockDim.x;
      const int i = e < d ? root_index(m, oy, ox, e) : -1;
      in[v] = i >= 0;
      am[v] = in[v] ? a[e] : 0.f;
      lo[v] = xl[in[v] ? i : 0];
      hi[v] = xh[in[v] ? i : 0];
    }
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      if (!in[v]) continue;
      if (CERT) s = __fadd_rd(s, fminf(__fmul_rd(am[v], lo[v]), __fmul_rd(am[v], hi[v])));
      else s += fminf(am[v] * lo[v], am[v] * hi[v]);
    }
  }
  float out;
  if (CERT) {
    s = block_fsum<1>(s, shf);
    out = __double2float_rd(__dsub_rd(__dadd_rd(cd[rl], (double)s), E[rl]));
  } else {
    s = block_sum(s, shf);
    out = cf[rl] + s;
  }
  if (threadIdx.x == 0) root_write(c, r, out);
}

// Unstable neurons (l < 0 < u) per property, one block each, eight neurons' loads in flight per thread
// (12,800 neurons: 48 us with one).
constexpr int COUNT_THREADS = 1024;
__global__ void __launch_bounds__(COUNT_THREADS) k_count_unstable(int H, const float* __restrict__ l,
                                                                  const float* __restrict__ u,
                                                                  int32_t* __restrict__ out) {
  __shared__ int tot;
  const int p = blockIdx.x;
  if (threadIdx.x == 0) tot = 0;
  __syncthreads();
  int n = 0;
  for (int j0 = threadIdx.x; j0 < H; j0 += 8 * COUNT_THREADS) {
    float lv[8], uv[8];
#pragma unroll
    for (int v = 0; v < 8; ++v) {
      const int j = j0 + v * COUNT_THREADS;
      lv[v] = j < H ? l[(size_t)p * H + j] : 0.f;
      uv[v] = j < H ? u[(size_t)p * H + j] : 0.f;
    }
#pragma unroll
    for (int v = 0; v < 8; ++v) n += lv[v] < 0.f && uv[v] > 0.f ? 1 : 0;
  }
  n = __reduce_add_sync(0xffffffffu, n);
  if ((threadIdx.x & 31) == 0) atomicAdd(&tot, n);
  __syncthreads();
  if (threadIdx.x == 0) out[p] = tot;
}

static int root_threads(int d) { return d >= 256 ? 256 : (d + 31) / 32 * 32; }

void launch_root_first(bool cert, const RootCtx& c, int P, const LayerGeom& g, const float* W, const float* b,
                       cudaStream_t s) {
  const long long total = (long long)P * g.d_out;
  if (total <= 0) return;
  const unsigned grid = (unsigned)((total * 32 + 255) / 256);
  if (cert) k_root_first<true><<<grid, 256, 0, s>>>(c, g, W, b, total);
  else k_root_first<false><<<grid, 256, 0, s>>>(c, g, W, b, total);
  ++g_launches;
}

void launch_root_top(const RootCtx& c, const LayerGeom& g, bool patch, const float* W, const float* b, float* A,
                     float* cf, double* cd, double* E, cudaStream_t s) {
  if (c.R <= 0) return;
  k_root_top<<<c.R, 128, 0, s>>>(c, g, patch ? 1 : 0, W, b, A, cf, cd, E);
  ++g_launches;
}

void launch_root_relax(bool cert, const RootCtx& c, const RootMap& m, int d, long long hoff, int rule,
                       float rule_value, const float* Ain, float* Lam, const float* bias, float* cf, double* cd,
                       double* E, const float* wm, double gamma, cudaStream_t s) {
  if (c.R <= 0) return;
  const int nt = root_threads(d);
  const uintptr_t mis = reinterpret_cast<uintptr_t>(Ain) | reinterpret_cast<uintptr_t>(Lam) |
                        reinterpret_cast<uintptr_t>(bias) | reinterpret_cast<uintptr_t>(c.l + hoff) |
                        reinterpret_cast<uintptr_t>(c.u + hoff) | (cert ? reinterpret_cast<uintptr_t>(wm + hoff) : 0);
  const bool vec = !m.n && d % 4 == 0 && c.H % 4 == 0 && (mis & 15) == 0;
  auto go = [&](auto* kernel) {
    kernel<<<c.R, nt, 0, s>>>(c, m, d, hoff, rule, rule_value, Ain, Lam, bias, cf, cd, E, wm, gamma);
  };
  if (cert && vec) go(k_root_relax<true, true>);
  else if (cert) go(k_root_relax<true, false>);
  else if (vec) go(k_root_relax<false, true>);
  else go(k_root_relax<false, false>);
  ++g_launches;
}

void launch_root_concretize(bool cert, const RootCtx& c, const RootMap& m, int d, const float* A0, const float* cf,
                            const double* cd, const double* E, cudaStream_t s) {
  if (c.R <= 0) return;
  const int nt = root_threads(d);
  if (cert) k_root_concretize<true><<<c.R, nt, 0, s>>>(c, m, d, A0, cf, cd, E);
  else k_root_concretize<false><<<c.R, nt, 0, s>>>(c, m, d, A0, cf, cd, E);
  ++g_launches;
}

void launch_count_unstable(int P, int H, const float* l, const float* u, int32_t* out, cudaStream_t s) {
  if (P <= 0 || !out) return;
  k_count_unstable<<<P, COUNT_THREADS, 0, s>>>(H, l, u, out);
  ++g_launches;
}

}  // namespace bcrown
