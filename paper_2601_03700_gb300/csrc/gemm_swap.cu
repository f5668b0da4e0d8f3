// Weight-streaming tcgen05 GEMM for sm_103a: C[M, N] = A[M, K] * W[N, K]^T with M <= 128 token rows.
//
// Such a pass reads every weight once and computes 2 M flops per weight: it is a stream over W.  The
// 128-token-row tile of gemm_tc.cu would load 128 operand rows per 32 to 256 weight rows, so its
// operand traffic is several times the weights'; the mma.sync kernels for at most 16 rows stage the
// whole operand in every CTA.  Here the weights are the M side of the MMA and the tokens its N side:
//
//  * A tile is 128 output features (the accumulator's lanes) x all token rows (its columns, 16 to
//    128). A stage holds KC k-chunks of 64: one 3-D TMA box of 128 weight rows and one of the token
//    rows, so that the operand costs NT / 128 of the weights in L2 reads and nothing in HBM.
//  * K of a tile is split over a thread-block cluster of up to 8 CTAs, as many as fill the GPU at two
//    CTAs per SM. The CTAs of a launch stream equal amounts and all are resident (or the launch is many
//    tiles long), so the stream needs no finer balance. After the main loop the cluster reduces and
//    scatters: the tile is cut into cells of 32 features x 32 tokens dealt out to the ranks, each rank
//    sends its partial sums of a cell to the cell's owner through distributed shared memory (over the
//    idle ring), and the owner adds them in rank order (the same sum every run) and applies the fused
//    epilogue. An earlier form (equal shares of all units, the last CTA to arrive at a tile adding the
//    others' partials from global memory) paid one L2 round trip per contributor and 32 tokens there:
//    16 to 27 us on GPT-2-small's layers of 33 tokens, where the whole product takes 8 to 10.
// Measured (kernel times without launch overlap), against the kernels that took these shapes: Llama-2-7B layers, 16 rows:
// SwiGLU input (180 MB) 54 -> 34 us, QKV with 8 K/V heads (50 MB) 42 -> 19, O and down (34 and 90 MB) 35 -> 18 on
// average, mapper FC2 / FC3 (537 MB) 204 / 182 -> 92 / 86 (79 at the measured HBM rate); 77 rows: 70 and 58 -> 21 to
// 46 us.
//  * Weights do not depend on the preceding kernel: the first stages' weights are issued before the
//    programmatic-dependent-launch wait, the token rows after it (not for the mapper's products in a
//    prompt pass: a layer that no token leaves has no rows, and its launch then must cost nothing).
//  * Every mbarrier wait is bounded, as in gemm_tc.cu; a CTA whose wait gives up still takes part in
//    the cluster's barriers, so its peers complete.
#define ADEPT_TU_ID 11
#include "gemm_swap.h"
#include "epilogue.cuh"
#include "gemm_tc.h"
#include "tc_ptx.cuh"

#include <algorithm>
#include <cstring>

namespace adept {
namespace {

constexpr int SW_BF = 128;                     // features per tile
constexpr int SW_BK = 64;                      // k per chunk: one 128-byte swizzle row
constexpr int SW_THREADS = 192;
constexpr int SW_W_CHUNK = SW_BF * SW_BK * 2;  // 16 KB
constexpr int SW_MAX_STAGES = 8;
constexpr int SW_MAX_SPLITS = 8;               // portable cluster size
constexpr int SW_CP = 36;                      // floats per feature row of a cell: 32 tokens, padded
constexpr int SW_CELL = 32 * SW_CP * 4;        // bytes of one rank's part of a cell
constexpr int SW_SMEM = 110 * 1024;            // dynamic shared memory of a CTA: two fit on an SM
constexpr long long SW_TIMEOUT_CYCLES = 4000000000LL;   // ~2 s at 2 GHz

struct SwGroup {
  CUtensorMap tw;   // W as {64, N, K / 64}, box {64, 128, KC}
  CUtensorMap tx;   // token rows as {64, rows, K / 64}, box {64, NT, KC}
  DevRange rows;
  int N, tiles, nks;
  Epi epi;
};

template <int MAXG>
struct SwParams {
  SwGroup g[MAXG];
  int n_groups;
  int nt;         // token rows per box (a multiple of 16)
  int tmem_cols;  // accumulator columns (nt rounded up to 32, then to a power of two)
  int stages;
  int splits;     // cluster size
  int apart;      // the cells' exchange has shared memory of its own at off_cells (0: over the ring)
  int off_cells;
  int ahead;      // weights before the dependency wait (not where there may well be no rows)
  unsigned* err;
  SpanCtx span;
};

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
// Four floats to the shared memory of the cluster's CTA `rank`, at this CTA's address `local`.
__device__ __forceinline__ void put_remote(uint32_t local, uint32_t rank, float a, float b, float c, float d) {
  asm volatile(
      "{\n.reg .b32 r;\nmapa.shared::cluster.u32 r, %0, %1;\nst.shared::cluster.v4.f32 [r], {%2, %3, %4, %5};\n}\n" ::"r"(
          local),
      "r"(rank), "f"(a), "f"(b), "f"(c), "f"(d)
      : "memory");
}

template <int KIND, int KC, int MAXG>
__global__ void __launch_bounds__(SW_THREADS) gemm_swap_kernel(const __grid_constant__ SwParams<MAXG> p) {
  KT_BEGIN();
  extern __shared__ uint8_t sw_smem_raw[];
  __shared__ __align__(8) uint64_t full[SW_MAX_STAGES], empty[SW_MAX_STAGES], accf;
  __shared__ uint32_t tmem_slot;
  __shared__ int s_abort, s_rb, s_M;
  __shared__ float s_bias[SW_BF];
  __shared__ long long s_cbase[KIND == EPI_QKV ? SW_MAX_ROWS : 1];   // cache epilogues: each row's slot, position
  __shared__ int s_pos[KIND == EPI_QKV ? SW_MAX_ROWS : 1];
  __shared__ unsigned s_span_left;
  __shared__ unsigned long long s_span_t0;
  SpanScope span(p.span, &s_span_left, &s_span_t0);

  const long long wlim = wait_limit();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  volatile int* abort_flag = &s_abort;
  uint8_t* smem = (uint8_t*)(((uintptr_t)sw_smem_raw + 1023) & ~(uintptr_t)1023);
  const int S = p.stages, nt = p.nt, splits = p.splits;
  const int x_chunk = nt * SW_BK * 2;
  const int stage_bytes = KC * (SW_W_CHUNK + x_chunk);

  // this CTA's problem, tile and part of K (the cluster's CTAs are consecutive)
  const int rank = (int)blockIdx.x % splits;
  int tile = (int)blockIdx.x / splits, gi = 0;
  while (gi + 1 < p.n_groups && tile >= p.g[gi].tiles) tile -= p.g[gi++].tiles;
  const SwGroup& g = p.g[gi];
  if (!p.ahead) {
    // nothing is read ahead: without rows the launch ends here
    pdl_wait();
    const int m = g.rows.e() - g.rows.b();
    if (m <= 0) return;   // (the whole cluster)
  }
  const int k_lo = (int)((long long)rank * g.nks / splits), n_st = (int)((long long)(rank + 1) * g.nks / splits) - k_lo;

  if (threadIdx.x == 0) {
    for (int s = 0; s < S; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    mbar_init(&accf, 1);
    s_abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  span.init();
  if (splits > 1 && p.apart) cluster_arrive();   // waited for before the exchange: every CTA has started
  if (warp == 1) {
    tmem_alloc(&tmem_slot, (uint32_t)p.tmem_cols);
    tmem_relinquish();
  }
  auto load_w = [&](int i, int s) {
    mbar_expect_tx(&full[s], (uint32_t)stage_bytes);
    tma_load_3d(&g.tw, &full[s], smem + s * stage_bytes, tile * SW_BF, (k_lo + i) * KC);
  };
  auto load_x = [&](int i, int s, int rb) {
    tma_load_3d(&g.tx, &full[s], smem + s * stage_bytes + KC * SW_W_CHUNK, rb, (k_lo + i) * KC);
  };
  const int pre = p.ahead ? min(S, n_st) : 0;   // the ring's weights before the wait
  if (threadIdx.x == 0)
    for (int i = 0; i < pre; ++i) load_w(i, i);
  pdl_wait();
  KT_WAITED();
  span.waited();
  if (threadIdx.x == 0) {
    const int b = g.rows.b();
    int M = max(0, g.rows.e() - b);
    if (M > nt) {                          // more rows than the launch was sized for
      atomicOr(p.err, ERRW_CONFIG);
      M = nt;
    }
    s_rb = b;
    s_M = M;
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  pdl_launch_dependents();   // after the TMEM allocation: a dependent CTA cannot take it first
  const int M = s_M, rb = s_rb;
  const uint32_t tmem = tmem_slot;
  // a wait for copies that this CTA has issued: they land whatever else happens
  auto land = [&](int s, uint32_t par) {
    const long long t0 = clock64();
    while (!mbar_try_wait(&full[s], par)) {
      if (clock64() - t0 > SW_TIMEOUT_CYCLES) {
        atomicOr(p.err, ERRW_TIMEOUT);
        break;
      }
    }
  };

  if (M == 0) {
    // no rows (the whole cluster sees none): the weights under way land (their stages complete with the token rows'
    // bytes), nothing else happens
    if (threadIdx.x == 0) {
      for (int i = 0; i < pre; ++i) load_x(i, i, rb);
      for (int i = 0; i < pre; ++i) land(i, 0);
    }
  } else {
    if (warp == 0) {
      if (elect_one()) {
        // ------------------------------------------------------------ TMA producer
        int s = 0, n = 0;   // slot and its use number
        uint32_t issued = 0, last_par = 0;
        for (int i = 0; i < n_st; ++i) {
          if (n > 0 && !mbar_wait(&empty[s], (uint32_t)((n - 1) & 1), abort_flag, p.err, wlim)) break;
          if (i >= pre) load_w(i, s);
          load_x(i, s, rb);
          issued |= 1u << s;
          last_par = (last_par & ~(1u << s)) | ((uint32_t)(n & 1) << s);
          if (++s == S) {
            s = 0;
            ++n;
          }
        }
        for (int k = 0; k < S; ++k)   // every copy has landed before the ring is used for the cells
          if (issued >> k & 1u) land(k, (last_par >> k) & 1u);
      }
    } else if (warp == 1) {
      if (elect_one()) {
        // ------------------------------------------------------------ MMA issuer
        // kind::f16: D fp32, A and B bf16, both K-major, M = 128, N = the live rows
        const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(((M + 15) >> 4) * 2) << 17) |
                               ((uint32_t)(SW_BF >> 4) << 24);
        int s = 0, n = 0;
        for (int i = 0; i < n_st; ++i) {
          if (!mbar_wait(&full[s], (uint32_t)(n & 1), abort_flag, p.err, wlim)) break;
          tc_fence_after();
          const uint32_t base = smem_u32(smem + s * stage_bytes);
#pragma unroll
          for (int k = 0; k < KC; ++k) {
            const uint64_t wd = sdesc_sw128(base + k * SW_W_CHUNK);
            const uint64_t xd = sdesc_sw128(base + KC * SW_W_CHUNK + k * x_chunk);
#pragma unroll
            for (int j = 0; j < SW_BK / 16; ++j)
              umma_bf16(tmem, wd + (uint64_t)(2 * j), xd + (uint64_t)(2 * j), idesc, (i | k | j) != 0 ? 1u : 0u);
          }
          umma_commit(&empty[s]);
          if (++s == S) {
            s = 0;
            ++n;
          }
        }
        // every MMA issued by this thread has completed: the accumulator is whole, TMEM may be freed
        umma_commit(&accf);
        const long long t0 = clock64();
        while (!mbar_try_wait(&accf, 0)) {
          if (clock64() - t0 > SW_TIMEOUT_CYCLES) {
            atomicOr(p.err, ERRW_TIMEOUT);
            break;
          }
        }
      }
    } else {
      // ------------- epilogue warps: what does not depend on the accumulator, while it fills
      const int et = (warp - 2) * 32 + lane, col = tile * SW_BF + et;
      s_bias[et] = (g.epi.bias && col < g.N) ? g.epi.bias[col] : 0.f;
      if (KIND == EPI_QKV && et < M) {
        const EpiRow rr = epi_row(g.epi, rb + et);
        s_cbase[et] = rr.cbase;
        s_pos[et] = rr.pos;
      }
    }
    __syncthreads();   // the accumulator is whole, the ring idle
    const bool ok = *abort_flag == 0;
    if (splits > 1) {   // ... in every CTA of the cluster, where the exchange goes over the ring
      if (!p.apart) cluster_arrive();
      cluster_wait();
    }
    tc_fence_after();
    // Cell (q, tb): features q * 32 .., tokens tb * 32 ..; number tb * 4 + q, owner number % splits. Its parts lie in the
    // owner's exchange as [number / splits][rank][feature][token].
    const int n_tb = (M + 31) >> 5;
    uint8_t* cells = smem + p.off_cells;
    if (warp >= 2) {
      const int q = warp & 3;   // TMEM lane quarter of this warp
      const uint32_t ta = tmem + ((uint32_t)(q * 32) << 16);
#pragma unroll 1
      for (int tb = 0; tb < n_tb; ++tb) {
        const int cell = tb * 4 + q, owner = cell % splits;
        float v[32];
        tmem_ld32(ta + (uint32_t)(tb * 32), v);
        const uint32_t at = smem_u32(cells) + (uint32_t)((cell / splits) * splits + rank) * SW_CELL + lane * SW_CP * 4;
#pragma unroll
        for (int j = 0; j < 8; ++j)
          put_remote(at + j * 16, (uint32_t)owner, v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
      }
    }
    if (splits > 1) {
      cluster_arrive();
      cluster_wait();
    } else {
      __syncthreads();
    }
    if (warp >= 2 && ok) {
      const int n_cells = n_tb * 4;
#pragma unroll 1
      for (int k = warp - 2; k * splits + rank < n_cells; k += 4) {
        const int cell = k * splits + rank, t = (cell >> 2) * 32 + lane, c0 = tile * SW_BF + (cell & 3) * 32;
        if (c0 >= g.N || t >= M) continue;
        const float* part = reinterpret_cast<const float*>(cells + (size_t)k * splits * SW_CELL) + lane;
        float o[32];
#pragma unroll
        for (int f = 0; f < 32; ++f) o[f] = part[f * SW_CP];
        for (int r = 1; r < splits; ++r) {
          part += SW_CELL / 4;
#pragma unroll
          for (int f = 0; f < 32; ++f) o[f] += part[f * SW_CP];
        }
        EpiRow rr{-1, 0, nullptr};
        if (KIND == EPI_QKV) {
          rr.cbase = s_cbase[t];
          rr.pos = s_pos[t];
        }
        epi_chunk32<bf16, KIND>(g.epi, rb + t, c0, g.N, o, rr, s_bias + (cell & 3) * 32);
      }
    }
    tc_fence_before();
  }
  __syncthreads();
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    tmem_dealloc(tmem, (uint32_t)p.tmem_cols);
  }
}

int g_sw_sms = 0;

template <int KIND, int KC, int MAXG>
int sw_launch(cudaStream_t st, const SwParams<MAXG>& prm, int grid, size_t smem) {
  static bool attr = false;
  if (!attr) {
    if (cudaFuncSetAttribute(gemm_swap_kernel<KIND, KC, MAXG>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             SW_SMEM) != cudaSuccess)
      return -1;
    attr = true;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(SW_THREADS);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = prm.splits;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = g_pdl ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, gemm_swap_kernel<KIND, KC, MAXG>, prm) == cudaSuccess ? 1 : -1;
}

template <int KC, int MAXG>
int sw_go(cudaStream_t st, const GemmProblem* probs, int n, int rows, unsigned* err) {
  thread_local SwParams<MAXG> prm;   // one per host thread
  memset(&prm, 0, sizeof prm);
  prm.n_groups = n;
  prm.nt = cdiv(rows, 16) * 16;
  prm.tmem_cols = 32;
  while (prm.tmem_cols < prm.nt) prm.tmem_cols *= 2;
  prm.ahead = 1;
  prm.err = err;
  prm.span = g_span;
  long long tiles = 0;
  int nks = 1 << 30, max_nks = 0;
  for (int i = 0; i < n; ++i) {
    const GemmProblem& q = probs[i];
    SwGroup& g = prm.g[i];
    if (!tc_encode_weight_3d(&g.tw, q.B, q.K, q.N, (size_t)q.ldb * 2, SW_BF, KC)) return -1;
    if (!tc_encode_weight_3d(&g.tx, q.A, q.K, q.a_rows, (size_t)q.lda * 2, prm.nt, KC)) return -1;
    g.rows = q.rows;
    g.N = q.N;
    g.tiles = cdiv(q.N, SW_BF);
    g.nks = cdiv(q.K, SW_BK * KC);
    g.epi = q.epi;
    if (q.split_live) prm.ahead = 0;
    tiles += g.tiles;
    nks = std::min(nks, g.nks);
    max_nks = std::max(max_nks, g.nks);
  }
  // as many CTAs per tile as fill the SMs twice, each with at least 3 k-chunks of 64 (12 at up to 16 rows): below
  // that the exchange costs more than the shorter loop saves (GPT-2-small prompt of 48 tokens, all layers: 785 us at
  // one chunk and more, 735 at 3, 755 at 4; of 16 tokens: 690 at 2, 669 at 4, 676 at 12, with exits 1039, 1010, 971)
  const int min_st = KC == 2 ? 6 : 3;
  prm.splits = (int)std::max(1LL, std::min<long long>({2LL * g_sw_sms / tiles, SW_MAX_SPLITS, nks / min_st}));
  const int stage = KC * (SW_W_CHUNK + prm.nt * SW_BK * 2);
  const int cells = cdiv(cdiv(prm.nt, 32) * 4, prm.splits) * prm.splits * SW_CELL;   // the exchange
  prm.stages = std::min({SW_MAX_STAGES, (SW_SMEM - 1024) / stage, std::max(2, cdiv(max_nks, prm.splits))});
  if (prm.stages < 2 || cells + 1024 > SW_SMEM || tiles * prm.splits > (1 << 30)) return -1;
  prm.apart = prm.stages * stage + cells + 1024 <= SW_SMEM;
  prm.off_cells = prm.apart ? prm.stages * stage : 0;
  const size_t smem = (size_t)(prm.apart ? prm.stages * stage + cells : std::max(prm.stages * stage, cells)) + 1024;
  const int grid = (int)tiles * prm.splits;
  if constexpr (MAXG > 2) {
    return sw_launch<EPI_QKV, KC, MAXG>(st, prm, grid, smem);   // several problems: cache epilogues
  } else {
    switch (probs[0].epi.kind) {
      case EPI_F32: return sw_launch<EPI_F32, KC, MAXG>(st, prm, grid, smem);
      case EPI_ACT: return sw_launch<EPI_ACT, KC, MAXG>(st, prm, grid, smem);
      case EPI_RESID: return sw_launch<EPI_RESID, KC, MAXG>(st, prm, grid, smem);
      case EPI_SWIGLU: return sw_launch<EPI_SWIGLU, KC, MAXG>(st, prm, grid, smem);
      default: return sw_launch<EPI_QKV, KC, MAXG>(st, prm, grid, smem);
    }
  }
}

}  // namespace

bool swap_gemm_supported(const GemmProblem& q, int max_rows) {
  if (max_rows < 1 || max_rows > SW_MAX_ROWS) return false;
  if (q.N <= 0 || q.K <= 0 || q.K % SW_BK || q.lda % 8 || q.ldb % 8 || q.a_rows <= 0) return false;
  if (((uintptr_t)q.A | (uintptr_t)q.B) & 15) return false;
  if ((q.epi.kind == EPI_QKV || q.epi.kind == EPI_KV || q.epi.kind == EPI_SWIGLU) && q.N % 32) return false;
  return q.epi.kind >= EPI_F32 && q.epi.kind <= EPI_KV;
}

int swap_gemm(cudaStream_t st, const GemmProblem* probs, int n_probs, const int* max_rows, unsigned* err) {
  if (n_probs < 1 || n_probs > SW_MAXG) return -1;
  int rows = 0;
  for (int i = 0; i < n_probs; ++i) {
    const GemmProblem& q = probs[i];
    if (!swap_gemm_supported(q, max_rows[i]) || q.epi.tile_stats) return -1;
    if (n_probs > 1 && q.epi.kind != EPI_QKV && q.epi.kind != EPI_KV) return -1;
    rows = std::max(rows, max_rows[i]);
  }
  if (!g_sw_sms) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&g_sw_sms, cudaDevAttrMultiProcessorCount, dev);
    if (g_sw_sms <= 0) g_sw_sms = 1;
  }
  // two k-chunks per stage (256 contiguous bytes of a weight row) while two stages and more fit
  if (rows <= 16)
    return n_probs <= 2 ? sw_go<2, 2>(st, probs, n_probs, rows, err)
                        : sw_go<2, SW_MAXG>(st, probs, n_probs, rows, err);
  return n_probs <= 2 ? sw_go<1, 2>(st, probs, n_probs, rows, err)
                      : sw_go<1, SW_MAXG>(st, probs, n_probs, rows, err);
}

ADEPT_KTRACE_ATTACH(sw)

ADEPT_WAIT_LIMIT_SETTER(sw)

}  // namespace adept
