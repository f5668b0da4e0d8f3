// fp32-FMA GEMMs: the path of the fp32 models, and the cross-check of the tensor-core GEMM.
// f32_rows_kernel (fp32, the epilogue fused) takes products of few rows (f32_rows_win);
// gemm_simt_kernel, a 64 x 64 tile with a separate epilogue pass, the rest and bf16 operands (its
// epilogue semantics are the reference for the fused tcgen05 epilogue).
#define ADEPT_TU_ID 2
#include "common.cuh"
#include "kernels.h"
#include "epilogue.cuh"

namespace adept {

// Whether f32_rows_kernel takes M rows of an N x K product, and not the 64 x 64 tiles.
//
// The rows kernel reads every weight again for each 8 rows and takes M N K / 6e12 s (above K = 8192, where a row's pieces leave L1
// between features, M N K / 3.6e12 s); the tiles take 0.18 us per element of K while they find a place on the SMs at once (about
// 120 tiles), then 1 / 608 of that more per tile. Up to K = 512 the launches weigh on the rows kernel (M N K / 4.6e12 s), and
// the tiles take 0.13 us. So the line is 1.1 or 0.6 million outputs for one turn of the tiles. Both sides measured over 29
// (N, K) from 256 x 256 to 32768 x 8192 and up to 256 rows: the better kernel is chosen in all but a few places near the
// line, and there it is within 13 %. At 64 and 128 rows, rows kernel / tiles in us: 4096 x 4096 197 / 738 and 370 / 715;
// 12288 x 4096 566 / 887 and 1118 / 989; 8192 x 16384 2499 / 3209 and 4994 / 3172; 32768 x 8192 3006 / 2081 and 5641 / 3634.
// Prompt of 256 rows, D = 4096, FFN 11008, 4 layers, mapper 8192 / 16384: 37.1 ms on the tiles alone, 44.9 on the rows
// kernel alone, 29.0 so; D = 1024 (mapper 4096 / 8192) 8.84, 5.35 and 5.02. Above 256 rows the tiles: of D = 1024, 512 rows
// took 8.53 ms on them and 9.20 on the rows kernel.
constexpr int F32_ROWS_MAX = 256;
__host__ __device__ inline bool f32_rows_win(int M, int N, int K) {
  if (M > F32_ROWS_MAX) return false;
  const long long line = K > 512 && K <= 8192 ? 1100000 : 600000;   // outputs M N, while the tiles take one turn
  const long long tiles = (long long)((N + 63) / 64) * ((M + 63) / 64), turn = 2432 + 5 * tiles;   // in 3040ths: 0.8 + tiles / 608
  return (long long)M * N * 3040 <= line * (turn > 3040 ? turn : 3040);
}

// C[r, n] = sum_k A[begin + r, k] * B[n, k] for the rows of the problem's range.
template <typename T>
__global__ void __launch_bounds__(256) gemm_simt_kernel(const T* __restrict__ A, int lda, const T* __restrict__ B,
                                                        int ldb, DevRange rows, int N, int K, float* C, int ldc,
                                                        int above) {
  PDL_ENTRY();
  __shared__ float As[16][64 + 1];
  __shared__ float Bs[16][64 + 1];
  const int rb = rows.b(), M = rows.e() - rb;
  if (above && f32_rows_win(M, N, K)) return;   // the rows kernel's
  const int m0 = blockIdx.y * 64, n0 = blockIdx.x * 64;
  if (m0 >= M) return;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  float acc[4][4] = {};
  for (int k0 = 0; k0 < K; k0 += 16) {
    for (int i = threadIdx.x; i < 1024; i += 256) {
      const int r = i >> 4, kk = i & 15, gk = k0 + kk;
      As[kk][r] = (m0 + r < M && gk < K) ? to_f(A[(size_t)(rb + m0 + r) * lda + gk]) : 0.f;
      Bs[kk][r] = (n0 + r < N && gk < K) ? to_f(B[(size_t)(n0 + r) * ldb + gk]) : 0.f;
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < 16; ++kk) {
      float a[4], b[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        a[i] = As[kk][ty * 4 + i];
        b[i] = Bs[kk][tx * 4 + i];
      }
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int r = m0 + ty * 4 + i;
    if (r >= M) continue;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int n = n0 + tx * 4 + j;
      if (n < N) C[(size_t)r * ldc + n] = acc[i][j];
    }
  }
}

// Epilogue of one output row (see EpiKind), one thread per 32-column chunk.
template <typename T>
__global__ void epilogue_kernel(Epi e, const float* __restrict__ C, int ldc, DevRange rows, int N, int above, int K) {
  PDL_ENTRY();
  const int rb = rows.b(), M = rows.e() - rb;
  const int r = blockIdx.x;
  if (r >= M || (above && f32_rows_win(M, N, K))) return;
  const int ra = rb + r;
  const float* c = C + (size_t)r * ldc;
  const EpiRow rr = epi_row(e, ra);
  for (int ch = threadIdx.x; ch * 32 < N; ch += blockDim.x) {
    const int c0 = ch * 32;
    float v[32];
#pragma unroll
    for (int j = 0; j < 32; ++j) v[j] = (c0 + j < N) ? c[c0 + j] : 0.f;
    epi_chunk32<T>(e, ra, c0, N, v, rr);
  }
}

// C[r, n] = sum_k A[r, k] * B[n, k] for a few rows, fp32, with the fused epilogue.
//
// The fp32 models are small: a product's weights lie in L2 and its time is latency. The 64 x 64 tile
// left most SMs idle (4 CTAs for 64 rows x 256 outputs) and walked K in 16-element steps with two
// barriers each, and its epilogue was a launch of its own. Here a warp takes 4 features x 8 rows with
// its lanes split over K: every weight of a 512-element slice of K is read once into registers, as
// float4 and before the programmatic-dependent-launch wait (`ahead`: the operand is a weight that no
// preceding kernel writes), so that after the wait only the rows are to come. WK warps of the CTA
// share a long K; the 32 sums of a warp meet by a transposing butterfly (31 shuffles, lane = sum).
// The tile of 4 * 8 / WK features x 8 rows goes through the epilogue one element per thread.
// Measured (tiny configuration: D = 256, FFN 1024, mapper 1024 / 2048; kernel times without launch overlap): one row
// 43 us a product on average plus 4 for its epilogue launch -> 2.3 to 5.0; its 64-token prompt and 16 steps 20.4 ->
// 2.0 ms.
constexpr int FR_THREADS = 256, FR_R = 8, FR_F = 4, FR_KC = 512;

template <int WK, int KIND>
__global__ void __launch_bounds__(FR_THREADS) f32_rows_kernel(const float* __restrict__ A, int lda,
                                                              const float* __restrict__ B, int ldb, DevRange rows,
                                                              int N, int K, Epi e, int ahead, int below) {
  KT_BEGIN();
  constexpr int WF = FR_THREADS / 32 / WK, FT = FR_F * WF;   // feature groups, features of the CTA
  constexpr int NJ = FR_KC / 128;                            // float4 per lane of a slice
  __shared__ float s_part[WK][FR_R][FT + 1];
  __shared__ float s_v[FR_R][FT + 1];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, wf = warp % WF, wk = warp / WF;
  // feature of the CTA's local index: consecutive, or (SwiGLU: gate and up rows interleaved in blocks
  // of 16) half of them gates and half the matching ups
  auto feature = [&](int lf) {
    if (KIND != EPI_SWIGLU || FT == 32) return (int)blockIdx.x * FT + lf;
    constexpr int PARTS = 32 / FT, H = FT / 2;
    const int block = blockIdx.x / PARTS, part = blockIdx.x % PARTS;
    return block * 32 + part * H + (lf < H ? lf : 16 + lf - H);
  };
  float4 w[FR_F][NJ];
  auto load_w = [&](int k0) {
#pragma unroll
    for (int f = 0; f < FR_F; ++f) {
      const int n = feature(wf * FR_F + f);
#pragma unroll
      for (int j = 0; j < NJ; ++j) {
        const int k = k0 + (j * 32 + lane) * 4;
        w[f][j] = n < N && k < K ? *reinterpret_cast<const float4*>(B + (size_t)n * ldb + k) : make_float4(0.f, 0.f, 0.f, 0.f);
      }
    }
  };
  if (ahead) load_w(wk * FR_KC);
  pdl_wait();
  KT_WAITED();
  pdl_launch_dependents();
  const int rb = rows.b(), M = rows.e() - rb, r0 = blockIdx.y * FR_R;
  if (r0 >= M || (below && !f32_rows_win(M, N, K))) return;   // (below: more rows are the tiles')
  const int nr = min(FR_R, M - r0);
  float acc[FR_F * FR_R];
#pragma unroll
  for (int i = 0; i < FR_F * FR_R; ++i) acc[i] = 0.f;
  for (int k0 = wk * FR_KC; k0 < K; k0 += WK * FR_KC) {
    if (!ahead || k0 >= WK * FR_KC) load_w(k0);
#pragma unroll
    for (int r = 0; r < FR_R; ++r) {
      if (r >= nr) break;
      const float* a = A + (size_t)(rb + r0 + r) * lda;
      float4 x[NJ];
#pragma unroll
      for (int j = 0; j < NJ; ++j) {
        const int k = k0 + (j * 32 + lane) * 4;
        x[j] = k < K ? *reinterpret_cast<const float4*>(a + k) : make_float4(0.f, 0.f, 0.f, 0.f);
      }
#pragma unroll
      for (int f = 0; f < FR_F; ++f)
#pragma unroll
        for (int j = 0; j < NJ; ++j) {
          float& c = acc[f * FR_R + r];
          c = fmaf(x[j].x, w[f][j].x, c);
          c = fmaf(x[j].y, w[f][j].y, c);
          c = fmaf(x[j].z, w[f][j].z, c);
          c = fmaf(x[j].w, w[f][j].w, c);
        }
    }
  }
  // lane i ends with sum i = (feature i >> 3, row i & 7)
#pragma unroll
  for (int o = 16; o; o >>= 1) {
    const bool up = lane & o;
#pragma unroll
    for (int i = 0; i < o; ++i) {
      const float give = up ? acc[i] : acc[i + o], keep = up ? acc[i + o] : acc[i];
      acc[i] = keep + __shfl_xor_sync(0xffffffffu, give, o);
    }
  }
  s_part[wk][lane & (FR_R - 1)][wf * FR_F + (lane >> 3)] = acc[0];
  __syncthreads();
  const int r = threadIdx.x / FT, lf = threadIdx.x % FT, ra = rb + r0 + r, c = feature(lf);
  const bool mine = r < nr && c < N;
  float v = 0.f;
  if (mine) {
#pragma unroll
    for (int k = 0; k < WK; ++k) v += s_part[k][r][lf];
    if (e.bias) v += e.bias[c];
  }
  if (KIND == EPI_SWIGLU || KIND == EPI_QKV) {   // the other member of a pair
    if (r < FR_R) s_v[r][lf] = v;
    __syncthreads();
  }
  if (!mine) return;
  if (KIND == EPI_F32) {
    e.out_f32[(size_t)ra * e.ld_f32 + c] = v;
  } else if (KIND == EPI_ACT) {
    v = apply_act(e.act, v);
    ((float*)e.out_t)[(size_t)ra * e.ld_t + c] = v;
    if (e.out_f32) e.out_f32[(size_t)ra * e.ld_f32 + c] = v;
  } else if (KIND == EPI_RESID) {
    e.out_f32[(size_t)ra * e.ld_f32 + c] = e.resid[(size_t)ra * e.ld_resid + c] + v;
  } else if (KIND == EPI_SWIGLU) {
    if ((c & 31) < 16)
      ((float*)e.out_t)[(size_t)ra * e.ld_t + (c >> 5) * 16 + (c & 15)] = silu_f(v) * s_v[r][lf + FT / 2];
  } else {   // EPI_QKV / EPI_KV: q -> out_t, k / v -> the row's cache slot; rotary pairs in adjacent features
    const EpiRow rr = epi_row(e, ra);
    const int dh = e.head_dim, half = dh >> 1, nq = e.n_q_cols, nkv = e.n_kv_cols;
    const int base = c < nq ? 0 : c < nq + nkv ? nq : nq + nkv, h = (c - base) / dh, d = (c - base) - h * dh;
    int od = d;
    if (e.rope && base < nq + nkv) {
      const int ip = d >> 1;
      const float2 cs = e.rope_table[(size_t)rr.pos * half + ip];
      const float o = s_v[r][lf ^ 1];
      // (x1, x2) -> (x1 cos - x2 sin, x2 cos + x1 sin)
      v = (d & 1) ? v * cs.x + o * cs.y : v * cs.x - o * cs.y;
      od = (d & 1) ? ip + half : ip;
    }
    if (c < nq)
      ((float*)e.out_t)[(size_t)ra * e.ld_t + h * dh + od] = v;
    else if (rr.cbase >= 0)
      ((float*)(c < nq + nkv ? e.cache.k : e.cache.v))[rr.cbase + (size_t)h * e.cache.head_stride() + od] = v;
  }
}

template <int WK>
static void f32_rows_go(cudaStream_t st, const GemmProblem& p, int max_rows, bool ahead, bool below) {
  constexpr int FT = FR_F * (FR_THREADS / 32 / WK);
  const dim3 grid(cdiv(p.N, FT), cdiv(max_rows, FR_R));
#define GO(KIND)                                                                                                  \
  launch_k(f32_rows_kernel<WK, KIND>, grid, FR_THREADS, 0, st, (const float*)p.A, p.lda, (const float*)p.B, p.ldb, \
           p.rows, p.N, p.K, p.epi, ahead ? 1 : 0, below ? 1 : 0)
  switch (p.epi.kind) {
    case EPI_F32: GO(EPI_F32); break;
    case EPI_ACT: GO(EPI_ACT); break;
    case EPI_RESID: GO(EPI_RESID); break;
    case EPI_SWIGLU: GO(EPI_SWIGLU); break;
    default: GO(EPI_QKV); break;   // EPI_KV: no query columns
  }
#undef GO
}

F32Rows gemm_f32_rows(cudaStream_t st, const GemmProblem& p, int max_rows, bool ahead) {
  if (max_rows < 1 || max_rows > F32_ROWS_MAX || p.N < 1 || p.K < 1) return F32_ROWS_NONE;
  if ((p.K | p.lda | p.ldb) % 4 || (((uintptr_t)p.A | (uintptr_t)p.B) & 15)) return F32_ROWS_NONE;
  if (p.epi.kind < EPI_F32 || p.epi.kind > EPI_KV) return F32_ROWS_NONE;
  if ((p.epi.kind == EPI_SWIGLU || p.epi.kind >= EPI_QKV) && p.N % 32) return F32_ROWS_NONE;
  // Every count up to max_rows (within 64 rows the largest decides: the tiles' time stands still), or only the count itself
  // where the host knows it. Otherwise the live count decides on the device: both kernels are launched, and the one whose count
  // it is not leaves at once (2 to 20 us on products of 0.5 ms and more). The weights are then not read ahead.
  bool all = f32_rows_win(max_rows, p.N, p.K);
  if (!p.rows.begin && !p.rows.end) {
    if (!all) return F32_ROWS_NONE;
  } else {
    for (int r = 64; r < max_rows; r += 64) all = all && f32_rows_win(r, p.N, p.K);
  }
  int most = max_rows;
  while (most > 1 && !f32_rows_win(most, p.N, p.K)) --most;
  // K slices of 512 over 1, 2 or 4 warps
  if (p.K <= FR_KC) f32_rows_go<1>(st, p, most, ahead && all, !all);
  else if (p.K <= 2 * FR_KC) f32_rows_go<2>(st, p, most, ahead && all, !all);
  else f32_rows_go<4>(st, p, most, ahead && all, !all);
  return all ? F32_ROWS_ALL : F32_ROWS_SOME;
}

void launch_gemm_simt(cudaStream_t st, int dt, const GemmProblem& p, int max_rows, float* scratch, bool above) {
  if (max_rows <= 0) return;
  dim3 grid(cdiv(p.N, 64), cdiv(max_rows, 64));
  const int up = above ? 1 : 0;
  if (dt == 1) {
    launch_k(gemm_simt_kernel<bf16>, grid, 256, 0, st, (const bf16*)p.A, p.lda, (const bf16*)p.B, p.ldb, p.rows, p.N, p.K,
                                                 scratch, p.N, up);
    launch_k(epilogue_kernel<bf16>, max_rows, 64, 0, st, p.epi, scratch, p.N, p.rows, p.N, up, p.K);
  } else {
    launch_k(gemm_simt_kernel<float>, grid, 256, 0, st, (const float*)p.A, p.lda, (const float*)p.B, p.ldb, p.rows, p.N,
                                                  p.K, scratch, p.N, up);
    launch_k(epilogue_kernel<float>, max_rows, 64, 0, st, p.epi, scratch, p.N, p.rows, p.N, up, p.K);
  }
}

extern "C" __attribute__((visibility("default"))) int adept_debug_f32_rows_win(int M, int N, int K) { return f32_rows_win(M, N, K); }

ADEPT_KTRACE_ATTACH(simt)

}  // namespace adept
