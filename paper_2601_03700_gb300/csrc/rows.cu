// Row-wise kernels of a pass whose work is moving rows: standardisation, the encoder's
// LayerNorm, and the exit step (test, compaction, moves) of passes above the register-resident
// generation-step kernel's size.
#define ADEPT_TU_ID 10
#include "common.cuh"
#include "kernels.h"
#include "row_group.cuh"

#include <algorithm>

namespace adept {

// All of them are bound by HBM / L2 traffic (a few fp32 row vectors per row), or by latency when
// the rows are few.  A row is held in registers as V float4 per thread, every load issued before
// the first reduction, by a group of TPR threads: a warp for rows of up to 1024 elements (no
// barrier in the reduction, eight rows per CTA), the whole CTA of 256 above.  V = 0: rows of more
// than 8192 elements, which are read again from memory after the reduction.
// (mean, 1 / deviation) of a row for the attention input of the family: two passes over the
// held row (the mean first), as the definition reads.  NORM_COPY: (0, 1).
template <int TPR, int V>
__device__ __forceinline__ float2 row_norm(const float4 (&x)[V ? V : 1], const float* src, bool vec, int sub, int D4,
                                           int D, int mode, float eps, float* red) {
  if (mode == NORM_COPY) return make_float2(0.f, 1.f);
  float mu[1] = {0.f};
  if (mode == NORM_LN) {
    if (V) {
#pragma unroll
      for (int j = 0; j < V; ++j)
        if (sub + j * TPR < D4) mu[0] += sum4(x[j]);
    } else {
      for (int v = sub; v < D4; v += TPR) mu[0] += sum4(row4(src, v, vec));
    }
    group_sum<TPR, 1>(mu, red);
    mu[0] /= D;
  }
  float s2[1] = {0.f};
  if (V) {
#pragma unroll
    for (int j = 0; j < V; ++j)
      if (sub + j * TPR < D4) {
        const float4 c = centre4(x[j], mu[0]);
        s2[0] += dot4(c, c);
      }
  } else {
    for (int v = sub; v < D4; v += TPR) {
      const float4 c = centre4(row4(src, v, vec), mu[0]);
      s2[0] += dot4(c, c);
    }
  }
  group_sum<TPR, 1>(s2, red);
  return make_float2(mu[0], rsqrtf(s2[0] / D + eps));
}

__device__ __forceinline__ float4 row4(const bf16* x, int v) {
  const uint2 u = reinterpret_cast<const uint2*>(x)[v];
  const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u.x));
  const float2 b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u.y));
  return make_float4(a.x, a.y, b.x, b.y);
}
__device__ __forceinline__ float4 row4(const float* x, int v) { return reinterpret_cast<const float4*>(x)[v]; }
__device__ __forceinline__ float4 add4(float4 a, float4 b) { return make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w); }

// Token (+ position, + type) embeddings into the residual stream X and, as the first attention's input, into xhat: standardised by
// smode, or for the encoder (family 2) both the LayerNorm with gain and shift. A token id outside [0, V) is flagged and reads row 0.
// 8192 rows of 768: 26 us with a CTA per row and an element per load, 14 so; 2048 of 4096 29 and 13. Few tokens (generation steps)
// take a CTA each.
template <typename T, int TPR, int V>
__global__ void __launch_bounds__(RW_THREADS)
    embed_rows_kernel(const int* __restrict__ tokens, int n_tok, const int* __restrict__ tok_pos, const T* __restrict__ E,
                      const T* __restrict__ P, const float* __restrict__ type_emb, const float* __restrict__ g,
                      const float* __restrict__ b, int family, int D, int vocab, float eps, float* __restrict__ X,
                      unsigned* err, T* __restrict__ xhat, int smode, float seps) {
  PDL_ENTRY();
  __shared__ float red[RW_THREADS / 32];
  constexpr int G = RW_THREADS / TPR;
  const int t = blockIdx.x * G + (int)threadIdx.x / TPR, sub = threadIdx.x & (TPR - 1), D4 = D >> 2;
  if (t >= n_tok) return;   // (a whole group)
  int tok = tokens[t];
  if (tok < 0 || tok >= vocab) {
    if (sub == 0) atomicOr(err, ERRW_TOKEN);
    tok = 0;
  }
  const int pos = P ? tok_pos[t] : 0;
  float4 x[V];
#pragma unroll
  for (int j = 0; j < V; ++j)
    if (sub + j * TPR < D4) x[j] = row4(E + (size_t)tok * D, sub + j * TPR);
  if (P) {
#pragma unroll
    for (int j = 0; j < V; ++j)
      if (sub + j * TPR < D4) x[j] = add4(x[j], row4(P + (size_t)pos * D, sub + j * TPR));
  }
  if (type_emb) {
#pragma unroll
    for (int j = 0; j < V; ++j)
      if (sub + j * TPR < D4) x[j] = add4(x[j], row4(type_emb, sub + j * TPR));
  }
  float* o = X + (size_t)t * D;
  T* oh = xhat + (size_t)t * D;
  const bool enc = family == 2;
  const float2 n = row_norm<TPR, V>(x, nullptr, true, sub, D4, D, enc ? (int)NORM_LN : smode, enc ? eps : seps, red);
#pragma unroll
  for (int j = 0; j < V; ++j) {
    const int v = sub + j * TPR;
    if (v >= D4) continue;
    float4 y = scale4(centre4(x[j], n.x), n.y);
    if (enc) {
      const float4 gg = row4(g, v), bb = row4(b, v);
      y = make_float4(y.x * gg.x + bb.x, y.y * gg.y + bb.y, y.z * gg.z + bb.z, y.w * gg.w + bb.w);
    }
    put4(o, v, enc ? y : x[j]);
    put4(oh, v, y);
  }
}

// Rows in_rows[r] (or r) of X standardised into row r of out.
template <typename T, int TPR, int V>
__global__ void __launch_bounds__(RW_THREADS)
    standardize_rows_kernel(const float* __restrict__ X, int ldx, const int* in_rows, DevRange rows, int D, int mode,
                            float eps, T* __restrict__ out, int ld_out, bool vec) {
  PDL_ENTRY();
  __shared__ float red[RW_THREADS / 32];
  constexpr int G = RW_THREADS / TPR;
  const int rb = rows.b(), re = rows.e(), D4 = D >> 2, sub = threadIdx.x & (TPR - 1);
  for (int r = rb + blockIdx.x * G + (int)threadIdx.x / TPR; r < re; r += gridDim.x * G) {
    const float* src = X + (size_t)(in_rows ? in_rows[r] : r) * ldx;
    float4 x[V ? V : 1];
#pragma unroll
    for (int j = 0; j < V; ++j)
      if (sub + j * TPR < D4) x[j] = row4(src, sub + j * TPR, vec);
    const float2 n = row_norm<TPR, V>(x, src, vec, sub, D4, D, mode, eps, red);
    T* o = out + (size_t)r * ld_out;
    if (V) {
#pragma unroll
      for (int j = 0; j < V; ++j)
        if (sub + j * TPR < D4) put4(o, sub + j * TPR, scale4(centre4(x[j], n.x), n.y));
    } else {
      for (int v = sub; v < D4; v += TPR) put4(o, v, scale4(centre4(row4(src, v, vec), n.x), n.y));
    }
  }
}

// The exit test of row r (token tok) from its sums |s_i|^2, |I|^2, <s_i, I>, |s_{i-1}|^2, <s_i, s_{i-1}>.
struct ExitTest {
  const int *row_tok, *forced;
  int layer, n_layers, test, metric;
  const float* delta;
  float* sim;
  int* flag;
  float* inv_norm;
  unsigned* err;
};
__device__ __forceinline__ void exit_decide(const ExitTest& t, int r, int tok, const float (&a)[5]) {
  int ex = 0;
  if (t.test) {
    const float c = exit_similarity(t.metric, a[0], a[1], a[2], a[3], a[4]);
    if (t.sim) t.sim[(size_t)tok * t.n_layers + (t.layer - 1)] = c;
    const int f = t.forced ? t.forced[tok] : 0;
    if (f != 0 && (f < 2 || f > t.n_layers)) atomicOr(t.err, ERRW_FORCED);
    ex = (f > 0) ? (f == t.layer) : (c >= *t.delta);
  }
  t.flag[r] = ex;
  t.inv_norm[r] = a[0] > 0.f ? rsqrtf(a[0]) : 0.f;
}

// The post-LN encoder's residual stream: LayerNorm with gain and shift in place, and the result
// as the next product's operand in the model's type (xt, optional, row stride D).
// TEST (V > 0): the layer's last LayerNorm, which also takes the exit test of the row while it is
// held (the test on its own read the row again and took a launch: 9.3 us for 8192 rows of 768).
template <typename T, int TPR, int V, bool TEST>
__global__ void __launch_bounds__(RW_THREADS)
    layernorm_rows_kernel(float* __restrict__ X, DevRange rows, int D, const float* __restrict__ g,
                          const float* __restrict__ b, float eps, T* __restrict__ xt, const float* __restrict__ I,
                          const float* __restrict__ Xin, ExitTest t) {
  PDL_ENTRY();
  __shared__ float red[RW_THREADS / 32 * (TEST ? 5 : 1)];
  constexpr int G = RW_THREADS / TPR;
  const int rb = rows.b(), re = rows.e(), D4 = D >> 2, sub = threadIdx.x & (TPR - 1);
  for (int r = rb + blockIdx.x * G + (int)threadIdx.x / TPR; r < re; r += gridDim.x * G) {
    float* src = X + (size_t)r * D;
    float4 x[V ? V : 1];
#pragma unroll
    for (int j = 0; j < V; ++j)
      if (sub + j * TPR < D4) x[j] = row4(src, sub + j * TPR, true);
    float4 c[TEST ? V : 1];
    if (TEST && t.test) {
#pragma unroll
      for (int j = 0; j < V; ++j)
        if (sub + j * TPR < D4) c[j] = row4(I + (size_t)r * D, sub + j * TPR, true);
    }
    const float2 n = row_norm<TPR, V>(x, src, true, sub, D4, D, NORM_LN, eps, red);
    auto out = [&](int v, float4 a) {
      const float4 c = scale4(centre4(a, n.x), n.y), gg = row4(g, v, true), bb = row4(b, v, true);
      const float4 y = make_float4(c.x * gg.x + bb.x, c.y * gg.y + bb.y, c.z * gg.z + bb.z, c.w * gg.w + bb.w);
      put4(src, v, y);
      if (xt) put4(xt + (size_t)r * D, v, y);
      return y;
    };
    if (V) {
      float a[5] = {0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int j = 0; j < V; ++j) {
        if (sub + j * TPR >= D4) continue;
        const float4 y = out(sub + j * TPR, x[j]);
        if (!TEST) continue;
        a[0] += dot4(y, y);
        if (t.test) {   // layer 1 tests nothing: only its norm is needed
          a[1] += dot4(c[j], c[j]);
          a[2] += dot4(y, c[j]);
          if (t.metric != EXIT_GLOBAL) {
            const float4 s = row4(Xin + (size_t)r * D, sub + j * TPR, true);
            a[3] += dot4(s, s);
            a[4] += dot4(y, s);
          }
        }
      }
      if (TEST) {
        group_sum<TPR, 5>(a, red);
        if (sub == 0) exit_decide(t, r, t.row_tok[r], a);
      }
    } else {
      for (int v = sub; v < D4; v += TPR) out(v, row4(src, v, true));   // a thread rewrites only what it reads
    }
  }
}

// ---------------------------------------------------------------------------
// exit test (Sec. 4.1): c = <s_i, I> / (|s_i| |I|) vs delta, or the forced layer
// ---------------------------------------------------------------------------
template <int TPR>
__global__ void __launch_bounds__(RW_THREADS)
    exit_decide_kernel(const float* __restrict__ Xout, const float* __restrict__ I, const float* __restrict__ Xin,
                       int D, DevRange rows, ExitTest t) {
  PDL_ENTRY();
  __shared__ float red[RW_THREADS / 32 * 5];
  const int r = blockIdx.x * (RW_THREADS / TPR) + (int)threadIdx.x / TPR, sub = threadIdx.x & (TPR - 1);
  if (r >= rows.e()) return;   // the whole group: with TPR = RW_THREADS the whole CTA
  const float4* s = reinterpret_cast<const float4*>(Xout + (size_t)r * D);
  const float4* in = reinterpret_cast<const float4*>(I + (size_t)r * D);
  const float4* sp = reinterpret_cast<const float4*>(Xin + (size_t)r * D);
  const int tok = t.row_tok[r];
  float a[5] = {0.f, 0.f, 0.f, 0.f, 0.f};   // |s_i|^2, |I|^2, <s_i, I>, |s_{i-1}|^2, <s_i, s_{i-1}>
  const int D4 = D >> 2;
#pragma unroll 4
  for (int v = sub; v < D4; v += TPR) {
    const float4 x = s[v];
    a[0] += dot4(x, x);
    if (t.test) {   // layer 1 tests nothing: only its norm is needed
      const float4 c = in[v];
      a[1] += dot4(c, c);
      a[2] += dot4(x, c);
      if (t.metric != EXIT_GLOBAL) {
        const float4 b = sp[v];
        a[3] += dot4(b, b);
        a[4] += dot4(x, b);
      }
    }
  }
  group_sum<TPR, 5>(a, red);
  if (sub != 0) return;
  exit_decide(t, r, tok, a);
}

// The compaction and the moves in one launch.  A CTA takes an equal run of the active rows; it
// counts the exits before its run (the flags are a few KB in L2) and places its own rows by a
// block scan, so that the stable order needs no launch of its own.  Survivors go to the next
// layer's input (s_i), their inertia with s_hat_i added (Sec. 4.1, after the test), and,
// standardised (smode, seps), to the next product's operand xhat; leaving rows to the mapper's
// input slots (s_i, s_{i-1}, inertia before s_hat_i).  first != 0 (layer 1): the inertia starts
// as s_hat_1 (the sum over earlier layers is empty).  Counters: ctr[CTR_ACTIVE + parity] active
// rows, ctr[CTR_PREFIX + i] exits after layer i, ctr[CTR_EXITED] exits so far; a CTA reads only
// counters that no CTA of the launch writes.
// Test and moves of 2048 rows x 4096: 27.8 (test) + 4.9 (scan) + 36 (moves) + 15.9 (standardise) ->
// 10.4 + 22.2 us, 151 MB moved at the HBM rate; of 8192 x 768: 9.0 + 9.8 + 16.3 + 8.0 -> 7.3 + 14.1.
// Passes of 17 to 256 rows, and of 5 to 16 rows of 4096, ran the whole step in one CTA before (470 us
// at 77 rows of 4096, 143 at 16): 12 us now.
// aao_len (all-at-once, = the prompt length): a row takes the decision of its sequence's last
// prompt token, which is active with it at the same row offset (sequences stay whole).
template <typename T, int TPR, int V>
__global__ void __launch_bounds__(RW_THREADS)
    exit_move_kernel(const float* __restrict__ Xin, const float* __restrict__ Xout, const float* __restrict__ I,
                     int first, int D, int* ctr, int par, const int* flag, const float* inv_norm, const int* row_tok,
                     int* row_tok_next, int* exit_tok, int* exit_layer_out, int layer, float* __restrict__ Xnext,
                     float* __restrict__ Inext, float* __restrict__ hsm_s, float* __restrict__ hsm_prev,
                     float* __restrict__ hsm_I, T* __restrict__ xhat, int smode, float seps, int aao_len,
                     const int* tok_pos) {
  PDL_ENTRY();
  __shared__ float red[RW_THREADS / 32];
  __shared__ int s_dst[RW_THREADS], s_cnt[RW_THREADS / 32];
  constexpr int G = RW_THREADS / TPR;
  const int n = ctr[CTR_ACTIVE + par], base = ctr[CTR_PREFIX + layer - 1];
  const int per = (n + gridDim.x - 1) / gridDim.x;
  const int lo = min(n, (int)blockIdx.x * per), hi = min(n, lo + per);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, sub = threadIdx.x & (TPR - 1), D4 = D >> 2;
  auto leaves = [&](int r) {
    return flag[aao_len ? min(n - 1, r + (aao_len - 1 - tok_pos[row_tok[r]])) : r];
  };
  if (n == 0) {
    if (blockIdx.x == 0 && threadIdx.x == 0) {
      ctr[CTR_ACTIVE + (par ^ 1)] = 0;
      ctr[CTR_EXITED] = base;
      ctr[CTR_PREFIX + layer] = base;
    }
    return;
  }
  if (lo >= hi) return;
  int before = 0;   // exits among the rows before this CTA's run
  for (int r = threadIdx.x; r < lo; r += RW_THREADS) before += leaves(r);
#pragma unroll
  for (int o = 16; o; o >>= 1) before += __shfl_xor_sync(0xffffffffu, before, o);
  if (lane == 0) s_cnt[warp] = before;
  __syncthreads();
  before = 0;
#pragma unroll
  for (int w = 0; w < RW_THREADS / 32; ++w) before += s_cnt[w];
  for (int b0 = lo; b0 < hi; b0 += RW_THREADS) {   // (one turn unless the pass is very large)
    const int m = min(RW_THREADS, hi - b0), r0 = b0 + (int)threadIdx.x;
    const bool mine = (int)threadIdx.x < m;
    const int tok = mine ? row_tok[r0] : 0;
    const bool ex = mine && leaves(r0) != 0;
    const unsigned bits = __ballot_sync(0xffffffffu, ex);
    __syncthreads();   // s_cnt and s_dst of the previous turn are read
    if (lane == 0) s_cnt[warp] = __popc(bits);
    __syncthreads();
    int e = before + __popc(bits & ((1u << lane) - 1u)), tot = 0;
#pragma unroll
    for (int w = 0; w < RW_THREADS / 32; ++w) {
      const int c = s_cnt[w];
      if (w < warp) e += c;
      tot += c;
    }
    if (mine) {
      if (ex) {
        s_dst[threadIdx.x] = -1 - (base + e);
        exit_tok[base + e] = tok;
        if (exit_layer_out) exit_layer_out[tok] = layer;
      } else {
        const int k = r0 - e;
        s_dst[threadIdx.x] = k;
        row_tok_next[k] = tok;
      }
    }
    before += tot;
    if (b0 + m == n && threadIdx.x == 0) {
      ctr[CTR_ACTIVE + (par ^ 1)] = n - before;
      ctr[CTR_EXITED] = base + before;
      ctr[CTR_PREFIX + layer] = base + before;
    }
    __syncthreads();
    for (int k = (int)threadIdx.x / TPR; k < m; k += G) {
      const int r = b0 + k, d0 = s_dst[k];
      const float* s = Xout + (size_t)r * D;
      const float* in = I + (size_t)r * D;
      if (d0 >= 0) {
        const float w = inv_norm[r];
        float* xn = Xnext + (size_t)d0 * D;
        float* inn = Inext + (size_t)d0 * D;
        T* xh = xhat + (size_t)d0 * D;
        float4 x[V ? V : 1], c[V ? V : 1];
#pragma unroll
        for (int j = 0; j < V; ++j)
          if (sub + j * TPR < D4) x[j] = row4(s, sub + j * TPR, true);
#pragma unroll
        for (int j = 0; j < V; ++j)
          if (sub + j * TPR < D4)
            c[j] = first ? make_float4(0.f, 0.f, 0.f, 0.f) : row4(in, sub + j * TPR, true);
        auto keep = [&](int v, float4 a, float4 i) {
          put4(xn, v, a);
          put4(inn, v, make_float4(i.x + a.x * w, i.y + a.y * w, i.z + a.z * w, i.w + a.w * w));
        };
        if (V) {
#pragma unroll
          for (int j = 0; j < V; ++j)
            if (sub + j * TPR < D4) keep(sub + j * TPR, x[j], c[j]);
        } else {
          for (int v = sub; v < D4; v += TPR)
            keep(v, row4(s, v, true), first ? make_float4(0.f, 0.f, 0.f, 0.f) : row4(in, v, true));
        }
        const float2 nm = row_norm<TPR, V>(x, s, true, sub, D4, D, smode, seps, red);
        if (V) {
#pragma unroll
          for (int j = 0; j < V; ++j)
            if (sub + j * TPR < D4) put4(xh, sub + j * TPR, scale4(centre4(x[j], nm.x), nm.y));
        } else {
          for (int v = sub; v < D4; v += TPR) put4(xh, v, scale4(centre4(row4(s, v, true), nm.x), nm.y));
        }
      } else {
        const size_t kk = (size_t)(-1 - d0) * D;
        const float* sp = Xin + (size_t)r * D;
#pragma unroll 2
        for (int v = sub; v < D4; v += TPR) {
          const float4 a = row4(s, v, true), b = row4(sp, v, true), c = row4(in, v, true);
          put4(hsm_s + kk, v, a);
          put4(hsm_prev + kk, v, b);
          put4(hsm_I + kk, v, c);
        }
      }
    }
  }
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
static int sm_count() {
  static const int sms = [] {
    int dev = 0, n = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    return std::max(n, 1);
  }();
  return sms;
}
// Grid of a kernel that takes its live rows (a device value) in turn, `per` rows at a time:
// enough CTAs for the row bound, at most four per SM.
static int rows_grid(int max_rows, int per) { return std::min(cdiv(max_rows, per), 4 * sm_count()); }

// GO(T, TPR, V) for a row of D elements (D is a multiple of 8).
#define ROWS_DISPATCH(T, D, GO)        \
  do {                                 \
    if ((D) <= 256) GO(T, 32, 2);      \
    else if ((D) <= 768) GO(T, 32, 6); \
    else if ((D) <= 1024) GO(T, 32, 8);\
    else if ((D) <= 4096) GO(T, 256, 4);\
    else if ((D) <= 8192) GO(T, 256, 8);\
    else GO(T, 256, 0);                \
  } while (0)

bool launch_embed_rows(cudaStream_t st, int dt, const int* tokens, int n_tok, const int* tok_pos, const void* E,
                       const void* P, const float* type_emb, const float* g, const float* b, int family, int D, int V,
                       float eps, float* X, unsigned* err, void* xhat, int smode, float seps) {
  if (D % 4 || D > 8192) return false;
  if (n_tok <= 0) return true;
#define GO(T, TPR, NV)                                                                                                \
  launch_k(embed_rows_kernel<T, TPR, NV>, cdiv(n_tok, RW_THREADS / TPR), RW_THREADS, 0, st, tokens, n_tok, tok_pos, \
           (const T*)E, (const T*)P, type_emb, g, b, family, D, V, eps, X, err, (T*)xhat, smode, seps)
#define PICK(T)                     \
  if (D <= 1024 && n_tok <= 16) GO(T, 256, 1); \
  else if (D <= 768) GO(T, 32, 6);  \
  else if (D <= 1024) GO(T, 32, 8); \
  else if (D <= 4096) GO(T, 256, 4); \
  else GO(T, 256, 8)
  if (dt == 1) {
    PICK(bf16);
  } else {
    PICK(float);
  }
#undef PICK
#undef GO
  return true;
}

void launch_standardize(cudaStream_t st, int dt, const float* X, int ldx, const int* in_rows, DevRange rows,
                        int max_rows, int D, int mode, float eps, void* out, int ld_out) {
  if (max_rows <= 0) return;
  // the library's own rows are 16-byte aligned; a caller's states may not be
  const bool vec = (uintptr_t)X % 16 == 0 && ldx % 4 == 0;
#define GO(T, TPR, V)                                                                                             \
  launch_k(standardize_rows_kernel<T, TPR, V>, rows_grid(max_rows, RW_THREADS / TPR), RW_THREADS, 0, st, X, ldx, \
           in_rows, rows, D, mode, eps, (T*)out, ld_out, vec)
  if (dt == 1) ROWS_DISPATCH(bf16, D, GO);
  else ROWS_DISPATCH(float, D, GO);
#undef GO
}

void launch_layernorm_rows(cudaStream_t st, int dt, float* X, DevRange rows, int max_rows, int D, const float* g,
                           const float* b, float eps, void* xt) {
  if (max_rows <= 0) return;
#define GO(T, TPR, V)                                                                                                    \
  launch_k(layernorm_rows_kernel<T, TPR, V, false>, rows_grid(max_rows, RW_THREADS / TPR), RW_THREADS, 0, st, X, rows, D, \
           g, b, eps, (T*)xt, (const float*)nullptr, (const float*)nullptr, ExitTest{})
  if (dt == 1) ROWS_DISPATCH(bf16, D, GO);
  else ROWS_DISPATCH(float, D, GO);
#undef GO
}

bool launch_layernorm_exit_test(cudaStream_t st, float* X, DevRange rows, int max_rows, int D, const float* g, const float* b,
                                float eps, const float* Xin, const float* I, const int* row_tok, const int* forced,
                                int layer, int n_layers, const float* delta_p, int test, int metric, float* sim, int* flag,
                                float* inv_norm, unsigned* err) {
  if (D > 8192) return false;   // (such rows are not held)
  if (max_rows <= 0) return true;
  const ExitTest t{row_tok, forced, layer, n_layers, test, metric, delta_p, sim, flag, inv_norm, err};
#define GO(T, TPR, V)                                                                                                     \
  launch_k(layernorm_rows_kernel<T, TPR, V ? V : 8, true>, rows_grid(max_rows, RW_THREADS / TPR), RW_THREADS, 0, st, X, rows, \
           D, g, b, eps, (T*)nullptr, I, Xin, t)
  ROWS_DISPATCH(float, D, GO);
#undef GO
  return true;
}

void launch_exit_rows(cudaStream_t st, int dt, const float* Xin, const float* Xout, const float* I, int first, int D,
                      int* ctr, int par, int max_rows, const int* row_tok, int* row_tok_next, const int* forced,
                      int layer, int n_layers, const float* delta_p, int test, int metric, float* sim, int* flag,
                      float* inv_norm, int* exit_tok, int* exit_layer_out, float* Xnext, float* Inext, float* hsm_s,
                      float* hsm_prev, float* hsm_I, void* xhat, int smode, float seps, int aao_len,
                      const int* tok_pos, unsigned* err, bool tested) {
  if (max_rows <= 0) return;
  const DevRange act{nullptr, ctr + CTR_ACTIVE + par, 0};
  const ExitTest t{row_tok, forced, layer, n_layers, test, metric, delta_p, sim, flag, inv_norm, err};
  if (tested) {
  } else if (D <= 1024) {
    launch_k(exit_decide_kernel<32>, cdiv(max_rows, RW_THREADS / 32), RW_THREADS, 0, st, Xout, I, Xin, D, act, t);
  } else {
    launch_k(exit_decide_kernel<256>, max_rows, RW_THREADS, 0, st, Xout, I, Xin, D, act, t);
  }
#define GO(T, TPR, V)                                                                                              \
  launch_k(exit_move_kernel<T, TPR, V>, rows_grid(max_rows, TPR == 32 ? 4 : 1), RW_THREADS, 0, st, Xin, Xout, I,   \
           first, D, ctr, par, flag, inv_norm, row_tok, row_tok_next, exit_tok, exit_layer_out, layer, Xnext, Inext, \
           hsm_s, hsm_prev, hsm_I, (T*)xhat, smode, seps, aao_len, tok_pos)
  if (dt == 1) ROWS_DISPATCH(bf16, D, GO);
  else ROWS_DISPATCH(float, D, GO);
#undef GO
}

ADEPT_KTRACE_ATTACH(rows)

}  // namespace adept
