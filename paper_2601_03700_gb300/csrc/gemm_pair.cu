// Grouped tcgen05 GEMM over CTA pairs for sm_103a: C[M, N] = A[M, K] * B[N, K]^T per problem (bf16 operands, both K-major;
// fp32 accumulation in tensor memory), one persistent launch over the tiles of every problem, fused epilogues.
//
//  * A tile is 256 rows x BN columns, computed by the two CTAs of a cluster with one cta_group::2 MMA: each CTA stages its
//    128 rows of A and half of the tile's B rows, so that an SM loads and the tensor core reads (128 + BN / 2) x 64 of
//    operands per k-block instead of (128 + BN) x 64.
//  * BN (32 to 256) is chosen by the kernel from the live row counts, which the host does not know (the rows that are still
//    active, or that leave, at a layer): the width whose whole waves of tiles take the least time. 2048 rows x 4096 outputs
//    are 2 full waves of 224 columns; in tiles of 256 they are 1.7. One launch serves every count.
//  * 8 epilogue warps per CTA (two per TMEM lane quarter, taking the tile's 32-column chunks in turn). A chunk leaves tensor
//    memory a row per lane and is turned around in shared memory, so that residuals and results move as whole 128-byte (bf16:
//    64-byte) row pieces; a row per lane took a transaction per lane. What a chunk needs besides the accumulator is read before
//    it, and the accumulator is given back by a relaxed arrive after its last read: a release at cluster scope waited for the
//    stores of the whole tile (8192 x 3072 x 768 with GELU 63 us, 45 without that wait). 12 or 16 warps leave a ring of 5
//    stages and too few registers: BERT-base 64 x 128 3.32 -> 3.53 and 3.58 ms, the 2048-token prompt 3.48 -> 3.68.
//
// Measured against the one-CTA tiles of 128 rows x 256 or 128 columns (gemm_tc.cu), which loaded 48 KB per k-block and SM (about
// 68 bytes per clock, the most seen) and ended in a last wave of a few tiles. 2048 rows: 12288 x 4096 144 -> 115 us (1.79
// PFLOP/s), 22016 x 4096 228 -> 200, 4096 x 11008 143 -> 105, 4096 x 4096 67 -> 50; 680 rows x 8192 x 32768 419 -> 259;
// 8192 rows x 768 x 768 with residual 36 -> 22, x 3072 x 768 with GELU 73 -> 45. Bound by the tensor cores from K of about 2000
// on (0.9 of their rate at the chosen width), by the epilogue's turn-around and stores below that.
//
// CTA = 10 warps: one thread of warp 0 TMA producer; warp 1 tensor-memory allocator, one of its threads in CTA 0 issues the pair's MMAs;
// warps 2..9 epilogue. Ring of k-blocks with full barriers in CTA 0 (both CTAs' copies complete on it) and empty barriers in
// both; two accumulator buffers. Waits are bounded: on time-out a CTA sets ERRW_TIMEOUT and stops; the pair leaves together, once
// every copy that either CTA issued has landed (pg_leave).
#define ADEPT_TU_ID 12
#include "gemm_pair.h"
#include "epilogue.cuh"
#include "gemm_tc.h"
#include "tc_ptx.cuh"

#include <algorithm>
#include <cstring>
#include <mutex>

namespace adept {
namespace {

constexpr int PG_BM = 256, PG_BK = 64;
constexpr int PG_EPI_WARPS = 8;
constexpr int PG_THREADS = 64 + 32 * PG_EPI_WARPS;
constexpr int PG_A_BYTES = 128 * PG_BK * 2;                 // a CTA's rows of A per k-block
constexpr int PG_RING = 6 * (PG_A_BYTES + 128 * PG_BK * 2); // 6 stages at BN = 256
constexpr int PG_MAX_STAGES = 10;
constexpr int PG_STG = 4096;                                // a warp's 32 x 32 fp32 chunk
constexpr int PG_SMEM = PG_RING + PG_EPI_WARPS * PG_STG + 1024;
// Candidate tile widths; a launch of many problems carries the tensor maps of every other one (its parameters have to fit
// a launch's 32 KB).
constexpr int PG_N_BN = 8;
constexpr int pg_step(int maxg) { return maxg <= 2 ? 1 : 2; }
constexpr int pg_width(int k) {
  return k == 0 ? 256 : k == 1 ? 224 : k == 2 ? 192 : k == 3 ? 160 : k == 4 ? 128 : k == 5 ? 96 : k == 6 ? 64 : 32;
}
constexpr long long PG_TIMEOUT_CYCLES = 4000000000LL;       // ~2 s at 2 GHz

template <int MAXG>
struct PgGroup {
  CUtensorMap ta;                             // A: box 64 x 128
  CUtensorMap tb[PG_N_BN / pg_step(MAXG)];    // B: box 64 x (half of each candidate width)
  DevRange rows;
  int N, K;
  int gm;             // m-tiles per raster super-row (their A rows stay in L2 while n sweeps)
  Epi epi;
};
template <int MAXG>
struct PgParams {
  PgGroup<MAXG> g[MAXG];
  int n_groups;
  unsigned* err;
};

__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// This CTA's shared-memory address `local` in CTA 0 of the pair.
__device__ __forceinline__ uint32_t at_leader(uint32_t local) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(r) : "r"(local));
  return r;
}
// Relaxed: it tells of accumulator reads (ordered by the tcgen05 fence before it) and of no memory; a release at cluster scope
// would wait for the warp's result stores.
__device__ __forceinline__ void arrive_cluster(uint32_t bar) {
  asm volatile("mbarrier.arrive.relaxed.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
// A 2-D box into this CTA's shared memory, completing on a barrier of either CTA of the pair.
__device__ __forceinline__ void pair_load_2d(const CUtensorMap* tm, uint32_t bar, uint32_t dst, int x, int y) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::
          "r"(dst),
      "l"((uint64_t)tm), "r"(x), "r"(y), "r"(bar));
}
__device__ __forceinline__ void pair_umma(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\ntcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
      "l"(a), "l"(b), "r"(idesc), "r"(accumulate)
      : "memory");
}
// Arrive on `bar` in both CTAs once every MMA issued so far by this thread has completed.
__device__ __forceinline__ void pair_commit(uint64_t* bar) {
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(smem_u32(bar)),
      "h"((uint16_t)3)
      : "memory");
}
__device__ __forceinline__ bool wait_fixed(uint64_t* bar, uint32_t par, unsigned* err) {
  const long long t0 = clock64();
  while (!mbar_try_wait(bar, par)) {
    if (clock64() - t0 > PG_TIMEOUT_CYCLES) {
      atomicOr(err, ERRW_TIMEOUT);
      return false;
    }
  }
  return true;
}

// A word to this CTA's shared-memory address `local` in the pair's other CTA.
__device__ __forceinline__ void put_peer(uint32_t local, int peer, uint32_t v) {
  asm volatile("{\n.reg .b32 r;\nmapa.shared::cluster.u32 r, %0, %1;\nst.shared::cluster.u32 [r], %2;\n}\n" ::"r"(local), "r"(peer),
               "r"(v)
               : "memory");
}
__device__ __forceinline__ int pg_stage_bytes(int bn) { return PG_A_BYTES + bn * (PG_BK * 2 / 2); }
__device__ __forceinline__ int pg_stages(int bn) { return min(PG_MAX_STAGES, PG_RING / pg_stage_bytes(bn)); }
// A pair that stopped early (every thread of both CTAs): waits until all copies that they issued have landed. Both CTAs' copies
// of a k-block complete on one barrier of CTA 0; a k-block that only one of them issued is given what the other did not send.
// Out of line: a register kept for it in the main loops is one too many.
__device__ __noinline__ void pg_leave(uint64_t* full, const uint32_t* issued, uint32_t* peer, int rank, int bn, unsigned* err) {
  if (threadIdx.x == 0) put_peer(smem_u32(peer), rank ^ 1, *issued);
  __syncwarp();
  cluster_sync_all();
  if (rank == 0 && threadIdx.x == 0) {
    const uint32_t n0 = *issued, n1 = *peer, stage_bytes = (uint32_t)pg_stage_bytes(bn);
    const int stages = pg_stages(bn);
    const long long t0 = clock64();
    bool ok = true;
    for (int s = 0; s < stages && ok; ++s) {
      const PgLanding l = pg_landing(n0, n1, (uint32_t)stages, (uint32_t)s);
      if (l.owe == PgLanding::NOTHING) continue;
      if (l.owe == PgLanding::ARRIVAL)
        mbar_expect_tx(&full[s], stage_bytes);
      else if (l.owe == PgLanding::BYTES)
        asm volatile("mbarrier.complete_tx.relaxed.cta.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&full[s])), "r"(stage_bytes) : "memory");
      while (ok && !mbar_try_wait(&full[s], l.parity)) ok = clock64() - t0 <= PG_TIMEOUT_CYCLES;
    }
    if (!ok) atomicOr(err, ERRW_TIMEOUT);
  }
  __syncwarp();
  cluster_sync_all();
}

// The time of one k-block of a tile in SM cycles: the MMAs take 2 BN (256 x BN x 64 at 8192 multiply-adds
// per clock and pair), the pair's SMs load (128 + BN / 2) x 128 bytes each at about 80 bytes per clock.
__device__ __forceinline__ float pg_block_cycles(int bn) { return fmaxf(2.f * bn, 205.f + 0.8f * bn); }

// ---------------------------------------------------------------------------- epilogue of one 32 x 32 chunk
// A staged chunk's rows lie one after another, their 16-byte pieces XOR-swizzled so that neither a piece per row (as tensor
// memory gives them) nor the pieces of whole rows (as they are read back) meet in a bank: fp32 rows of 8 pieces, bf16 rows of
// 4, SwiGLU's 16 bf16 results in 2.
__device__ __forceinline__ int piece32(int r, int p) { return r * 128 + ((p ^ (r & 7)) << 4); }
__device__ __forceinline__ int piece16(int r, int p) { return r * 64 + ((p ^ ((r >> 1) & 3)) << 4); }
__device__ __forceinline__ int piece8(int r, int p) { return r * 32 + ((p ^ ((r >> 2) & 1)) << 4); }
__device__ __forceinline__ uint32_t bf16x2(float a, float b) {
  const __nv_bfloat162 x = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<const uint32_t*>(&x);
}
// bf_only: the results are rounded to bf16 and kept in no wider type
__device__ __forceinline__ void act32(int act, bool bf_only, float (&v)[32]) {
  if (act == ACT_GELU_ERF && bf_only) {
#pragma unroll
    for (int j = 0; j < 32; ++j) v[j] = gelu_erf_bf(v[j]);
  } else {
    act_chunk32<bf16>(act, v);
  }
}

// Whether the chunk epilogues may move 16-byte pieces of the operands they use.
template <int KIND>
__device__ __forceinline__ bool pg_vectors(const Epi& e) {
  const bool f32 = ((uintptr_t)e.out_f32 & 15) == 0 && (e.ld_f32 & 3) == 0, t = ((uintptr_t)e.out_t & 15) == 0 && (e.ld_t & 7) == 0;
  switch (KIND) {
    case EPI_F32: return f32;
    case EPI_ACT: return t && (!e.out_f32 || f32);
    case EPI_RESID: return f32 && (!e.resid || (((uintptr_t)e.resid & 15) == 0 && (e.ld_resid & 3) == 0));
    case EPI_SWIGLU: return t;
    default: return true;   // heads of whole 32-column chunks
  }
}

// The epilogue of 32 rows of a tile.
template <int KIND>
struct PgTile {
  const Epi& e;
  uint8_t* stg;        // the warp's staging chunk
  int lane, ra0, n_rows, cb, ce, N;   // rows ra0 .., columns cb .. cb + ce
  bool vec;
  EpiRow rr;           // cache epilogues: this lane's row
  // what a chunk reads besides the accumulator
  struct In {
    float bias;        // of column `lane`
    float4 rs[KIND == EPI_RESID ? 8 : 1];
  };

  __device__ __forceinline__ void load(In& in, int c) const {
    const int lr = lane >> 3, lp = lane & 7, c0 = cb + c;
    if (c >= ce) return;
    in.bias = (e.bias && c0 + lane < N) ? e.bias[c0 + lane] : 0.f;
    if (KIND == EPI_RESID && !e.resid) {
#pragma unroll
      for (int i = 0; i < 8; ++i) in.rs[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    } else if (KIND == EPI_RESID && vec && c0 + 32 <= N) {
      const float* src = e.resid + (size_t)(ra0 + lr) * e.ld_resid + c0 + lp * 4;
      const size_t step = (size_t)4 * e.ld_resid;
#pragma unroll
      for (int i = 0; i < 8; ++i, src += step)
        in.rs[i] = 4 * i + lr < n_rows ? *reinterpret_cast<const float4*>(src) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
  }
  __device__ __forceinline__ float4 staged32(int r, int p) const { return *reinterpret_cast<const float4*>(stg + piece32(r, p)); }
  __device__ __forceinline__ void stage32(const float (&v)[32]) const {
#pragma unroll
    for (int k = 0; k < 8; ++k)
      *reinterpret_cast<float4*>(stg + piece32(lane, k)) = make_float4(v[4 * k], v[4 * k + 1], v[4 * k + 2], v[4 * k + 3]);
    __syncwarp();
  }
  __device__ __forceinline__ void stage16(const float (&v)[32]) const {
#pragma unroll
    for (int k = 0; k < 4; ++k)
      *reinterpret_cast<uint4*>(stg + piece16(lane, k)) =
          make_uint4(bf16x2(v[8 * k], v[8 * k + 1]), bf16x2(v[8 * k + 2], v[8 * k + 3]), bf16x2(v[8 * k + 4], v[8 * k + 5]),
                     bf16x2(v[8 * k + 6], v[8 * k + 7]));
    __syncwarp();
  }
  // F32 / ACT / RESID chunks with a ragged edge, or whose rows are not whole pieces: a lane per column, a row at a time.
  __device__ __forceinline__ void store_columns(int c0) const {
    const int c = c0 + lane;
#pragma unroll 1
    for (int r = 0; r < n_rows; ++r) {
      const float v = *reinterpret_cast<const float*>(stg + piece32(r, lane >> 2) + (lane & 3) * 4);
      if (c >= N) continue;
      const size_t ra = (size_t)(ra0 + r);
      if (KIND == EPI_ACT) ((bf16*)e.out_t)[ra * e.ld_t + c] = from_f<bf16>(v);
      if (KIND != EPI_ACT || e.out_f32)
        e.out_f32[ra * e.ld_f32 + c] = KIND == EPI_RESID && e.resid ? v + e.resid[ra * e.ld_resid + c] : v;
    }
  }
  // 32 fp32 results per row, with the residual: a row piece of 128 bytes per 8 lanes
  __device__ __forceinline__ void store32(int c0, const In& in) const {
    const int lr = lane >> 3, lp = lane & 7;
    float* o = e.out_f32 + (size_t)(ra0 + lr) * e.ld_f32 + c0 + lp * 4;
    const size_t step = (size_t)4 * e.ld_f32;
#pragma unroll
    for (int i = 0; i < 8; ++i, o += step) {
      float4 y = staged32(4 * i + lr, lp);
      if (KIND == EPI_RESID) y = make_float4(y.x + in.rs[i].x, y.y + in.rs[i].y, y.z + in.rs[i].z, y.w + in.rs[i].w);
      if (4 * i + lr < n_rows) *reinterpret_cast<float4*>(o) = y;
    }
  }

  // free: the pair's barrier for this accumulator, told after the warp's last read of it
  __device__ __forceinline__ void chunk(uint32_t tb, int c, const In& in, uint32_t free, bool last) const {
    const int c0 = cb + c;
    float v[32];
    tmem_ld32(tb + (uint32_t)c, v);
    tc_fence_before();
    __syncwarp();   // the chunk before this one has been read
    if (last && lane == 0) arrive_cluster(free);
    if (e.bias) {
      reinterpret_cast<float*>(stg)[lane] = in.bias;
      __syncwarp();
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const float4 b = reinterpret_cast<const float4*>(stg)[k];
        v[4 * k] += b.x;
        v[4 * k + 1] += b.y;
        v[4 * k + 2] += b.z;
        v[4 * k + 3] += b.w;
      }
      __syncwarp();
    }
    if constexpr (KIND == EPI_SWIGLU) {
      // the row's 16 gate and 16 up columns meet in this lane
#pragma unroll
      for (int j = 0; j < 16; ++j) v[j] = silu_f(v[j]) * v[16 + j];
#pragma unroll
      for (int k = 0; k < 2; ++k)
        *reinterpret_cast<uint4*>(stg + piece8(lane, k)) =
            make_uint4(bf16x2(v[8 * k], v[8 * k + 1]), bf16x2(v[8 * k + 2], v[8 * k + 3]), bf16x2(v[8 * k + 4], v[8 * k + 5]),
                       bf16x2(v[8 * k + 6], v[8 * k + 7]));
      __syncwarp();
      const int lr = lane >> 1, lp = lane & 1;
      bf16* o = (bf16*)e.out_t + (size_t)(ra0 + lr) * e.ld_t + (c0 >> 1) + lp * 8;
#pragma unroll
      for (int i = 0; i < 2; ++i, o += (size_t)16 * e.ld_t) {
        if (16 * i + lr >= n_rows) continue;
        const uint4 x = *reinterpret_cast<const uint4*>(stg + piece8(16 * i + lr, lp));
        if (vec) {
          *reinterpret_cast<uint4*>(o) = x;
        } else {
          const bf16* h = reinterpret_cast<const bf16*>(&x);
#pragma unroll
          for (int j = 0; j < 8; ++j) o[j] = h[j];
        }
      }
    } else if constexpr (KIND <= EPI_RESID) {
      if (KIND == EPI_ACT) act32(e.act, e.out_f32 == nullptr, v);
      const bool whole = vec && c0 + 32 <= N;
      if (KIND != EPI_ACT || !whole || e.out_f32) {
        stage32(v);
        if (!whole) {
          store_columns(c0);
          return;
        }
        store32(c0, in);
      }
      if constexpr (KIND == EPI_ACT) {
        if (e.out_f32) __syncwarp();
        stage16(v);
        const int lr = lane >> 2, lp = lane & 3;
        bf16* o = (bf16*)e.out_t + (size_t)(ra0 + lr) * e.ld_t + c0 + lp * 8;
        const size_t step = (size_t)8 * e.ld_t;
#pragma unroll
        for (int i = 0; i < 4; ++i, o += step)
          if (8 * i + lr < n_rows) *reinterpret_cast<uint4*>(o) = *reinterpret_cast<const uint4*>(stg + piece16(8 * i + lr, lp));
      }
    } else {
      // query columns, then key, then value (a chunk lies inside one head of one of them)
      const int dh = e.head_dim, nq = e.n_q_cols, nkv = e.n_kv_cols, lr = lane >> 2, lp = lane & 3;
      const bool is_q = c0 < nq, is_k = !is_q && c0 < nq + nkv;
      const int cc = is_q ? c0 : is_k ? c0 - nq : c0 - nq - nkv, h = cc / dh, d0 = cc - h * dh;
      bf16* base = is_q ? (bf16*)e.out_t + (size_t)ra0 * e.ld_t + h * dh
                        : (bf16*)(is_k ? e.cache.k : e.cache.v) + (size_t)h * e.cache.head_stride();
      const bool rope = e.rope && (is_q || is_k);
      if (rope)
        stage32(v);
      else
        stage16(v);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int r = 8 * i + lr;
        long long slot = __shfl_sync(0xffffffffu, rr.cbase, r);
        const int pos = __shfl_sync(0xffffffffu, rr.pos, r);
        if (is_q) slot = (long long)r * e.ld_t;
        if (r >= n_rows || slot < 0) continue;
        if (rope) {
          // columns (2 j, 2 j + 1) hold the rotate-half pair (j, j + dh / 2); 4 pairs per lane
          const int half_d = dh >> 1, j0 = (d0 >> 1) + lp * 4;
          const float4* tab = reinterpret_cast<const float4*>(e.rope_table + (size_t)pos * half_d + j0);
          const float4 x = staged32(r, 2 * lp), y = staged32(r, 2 * lp + 1), s = tab[0], t = tab[1];
          bf16* d = base + slot + j0;
          const float2 a0 = rope_turn(x.x, x.y, s.x, s.y), a1 = rope_turn(x.z, x.w, s.z, s.w);
          const float2 a2 = rope_turn(y.x, y.y, t.x, t.y), a3 = rope_turn(y.z, y.w, t.z, t.w);
          *reinterpret_cast<uint2*>(d) = make_uint2(bf16x2(a0.x, a1.x), bf16x2(a2.x, a3.x));
          *reinterpret_cast<uint2*>(d + half_d) = make_uint2(bf16x2(a0.y, a1.y), bf16x2(a2.y, a3.y));
        } else {
          *reinterpret_cast<uint4*>(base + slot + d0 + lp * 8) = *reinterpret_cast<const uint4*>(stg + piece16(r, lp));
        }
      }
    }
  }
};

// ---------------------------------------------------------------------------- kernel
// KIND: the epilogue of every problem of the launch (EPI_QKV also for EPI_KV, EPI_RESID also for EPI_F32)
template <int KIND, int MAXG>
__global__ void __launch_bounds__(PG_THREADS, 1) gemm_pair_kernel(const __grid_constant__ PgParams<MAXG> p) {
  KT_BEGIN();
  extern __shared__ uint8_t pg_smem_raw[];
  __shared__ __align__(8) uint64_t full[PG_MAX_STAGES], empty[PG_MAX_STAGES], accf[2], acce[2], drain;
  __shared__ uint32_t tmem_slot;
  __shared__ int s_abort, s_bn, s_map;
  __shared__ uint32_t s_issued, s_peer, s_stop;   // k-blocks whose copies this CTA issued; the other's; the other stopped early
  __shared__ int s_tile0[MAXG + 1], s_mbeg[MAXG], s_M[MAXG];

  const long long wlim = wait_limit();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = (int)(blockIdx.x & 1), pair = (int)(blockIdx.x >> 1), n_pairs = (int)(gridDim.x >> 1);
  const int ng = p.n_groups;
  volatile int* abort_flag = &s_abort;
  uint8_t* smem = (uint8_t*)(((uintptr_t)pg_smem_raw + 1023) & ~(uintptr_t)1023);

  // nothing here touches what an earlier kernel writes
  if (threadIdx.x == 0) {
    for (int s = 0; s < PG_MAX_STAGES; ++s) {
      mbar_init(&full[s], 1);    // CTA 0's producer; the bytes of both CTAs
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&accf[b], 1);
      mbar_init(&acce[b], 2 * PG_EPI_WARPS);
    }
    mbar_init(&drain, 1);
    s_abort = 0;
    s_issued = s_stop = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"((uint64_t)&p.g[0].ta) : "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)), "r"(512u)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  pdl_wait();
  KT_WAITED();
  if (warp == 0) {
    // live rows of the groups (a lane each); tile width (a lane per candidate); first tile of each group
    int M = 0;
    if (lane < ng) {
      const int b = p.g[lane].rows.b();
      M = max(0, p.g[lane].rows.e() - b);
      s_mbeg[lane] = b;
      s_M[lane] = M;
    }
    __syncwarp();
    constexpr int STEP = pg_step(MAXG), N_BN = PG_N_BN / STEP;
    const int bn = pg_width((lane & (N_BN - 1)) * STEP);
    int tiles = 0;
    float blocks = 0.f;   // k-blocks of all tiles
    for (int g = 0; g < ng; ++g) {
      const int t = ((s_M[g] + PG_BM - 1) >> 8) * ((p.g[g].N + bn - 1) / bn);
      tiles += t;
      blocks += (float)t * (float)((p.g[g].K + PG_BK - 1) / PG_BK);
    }
    float cost = 0.f;   // whole waves x (k-loop + what does not overlap the next tile)
    if (tiles > 0)
      cost = (float)((tiles + n_pairs - 1) / n_pairs) * (blocks / (float)tiles * pg_block_cycles(bn) + 200.f) + 12.f * bn;
    int best = lane & (N_BN - 1);
#pragma unroll
    for (int o = N_BN / 2; o; o >>= 1) {
      const float oc = __shfl_xor_sync(0xffffffffu, cost, o);
      const int ob = __shfl_xor_sync(0xffffffffu, best, o);
      if (oc < cost || (oc == cost && ob < best)) {
        cost = oc;
        best = ob;
      }
    }
    const int BN = pg_width(best * STEP);
    const int mine = lane < ng ? ((M + PG_BM - 1) >> 8) * ((p.g[lane].N + BN - 1) / BN) : 0;
    int sum = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int x = __shfl_up_sync(0xffffffffu, sum, o);
      if (lane >= o) sum += x;
    }
    if (lane < ng) s_tile0[lane + 1] = sum;
    if (lane == 0) {
      s_tile0[0] = 0;
      s_bn = BN;
      s_map = best;
    }
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();   // both CTAs' barriers and tensor memory are ready
  tc_fence_after();
  pdl_launch_dependents();
  const int BN = s_bn, total = s_tile0[ng];
  const uint32_t tmem = tmem_slot;
  const int stage_bytes = pg_stage_bytes(BN);
  const int S = pg_stages(BN);

  // Tile order inside a problem: super-rows of gm m-tiles; within one n is the outer and m the inner index.
  auto locate = [&](int t, int& g, int& mb, int& nb) {
    g = 0;
    while (g + 1 < ng && t >= s_tile0[g + 1]) ++g;
    const int local = t - s_tile0[g];
    const int tn = (p.g[g].N + BN - 1) / BN, tm = (s_M[g] + PG_BM - 1) >> 8, gm = p.g[g].gm;
    const int sup = local / (gm * tn), rem = local - sup * gm * tn, rows = min(gm, tm - sup * gm);
    nb = rem / rows;
    mb = sup * gm + rem % rows;
  };

  if (pair < total) {   // (uniform over the pair)
    if (warp == 0) {
      if (elect_one()) {
        // ------------------------------------------------------------ TMA producer (both CTAs)
        const uint32_t smem0 = smem_u32(smem), full0 = at_leader(smem_u32(full));
        int s = 0;
        uint32_t ph = 0, n_issued = 0;
        bool ok = true;
        for (int t = pair; t < total && ok; t += n_pairs) {
          int g, mb, nb;
          locate(t, g, mb, nb);
          const PgGroup<MAXG>& G = p.g[g];
          const int nk = (G.K + PG_BK - 1) / PG_BK;
          const int ya = s_mbeg[g] + mb * PG_BM + rank * 128, yb = nb * BN + rank * (BN / 2);
          const CUtensorMap *ta = &G.ta, *tb = &G.tb[s_map];
          for (int kb = 0; kb < nk; ++kb) {
            if (n_issued >= (uint32_t)S && !(ok = mbar_wait(&empty[s], ph ^ 1, abort_flag, p.err, wlim))) break;
            ++n_issued;
            const uint32_t bar = full0 + (uint32_t)s * 8;
            if (rank == 0) mbar_expect_tx(&full[s], (uint32_t)(2 * stage_bytes));
            const uint32_t dst = smem0 + (uint32_t)(s * stage_bytes);
            pair_load_2d(ta, bar, dst, kb * PG_BK, ya);
            pair_load_2d(tb, bar, dst + PG_A_BYTES, kb * PG_BK, yb);
            if (++s == S) {
              s = 0;
              ph ^= 1;
            }
          }
        }
        s_issued = n_issued;
      }
    } else if (warp == 1) {
      if (rank == 0 && elect_one()) {
        // ------------------------------------------------------------ MMA issuer (CTA 0)
        // kind::f16: D fp32, A and B bf16, both K-major, M = 256, N = BN
        const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(BN >> 3) << 17) | ((uint32_t)(PG_BM >> 4) << 24);
        const uint32_t smem0 = smem_u32(smem);
        int s = 0, ab = 0;
        uint32_t ph = 0, aph = 0;
        bool ok = true;
        for (int t = pair; t < total && ok; t += n_pairs) {
          int g, mb, nb;
          locate(t, g, mb, nb);
          const int nk = (p.g[g].K + PG_BK - 1) / PG_BK;
          if (!(ok = mbar_wait(&acce[ab], aph ^ 1, abort_flag, p.err, wlim))) break;
          tc_fence_after();
          const uint32_t d = tmem + (uint32_t)(ab * 256);
          for (int kb = 0; kb < nk; ++kb) {
            if (!(ok = mbar_wait(&full[s], ph, abort_flag, p.err, wlim))) break;
            tc_fence_after();
            const uint64_t ad = sdesc_sw128(smem0 + (uint32_t)(s * stage_bytes));
            const uint64_t bd = sdesc_sw128(smem0 + (uint32_t)(s * stage_bytes) + PG_A_BYTES);
#pragma unroll
            for (int k = 0; k < PG_BK / 16; ++k)
              pair_umma(d, ad + (uint64_t)(2 * k), bd + (uint64_t)(2 * k), idesc, (kb | k) != 0 ? 1u : 0u);
            pair_commit(&empty[s]);
            if (++s == S) {
              s = 0;
              ph ^= 1;
            }
          }
          if (!ok) break;
          pair_commit(&accf[ab]);
          ab ^= 1;
          if (ab == 0) aph ^= 1;
        }
        pair_commit(&drain);   // in both CTAs: no MMA reads their shared memory or writes their tensor memory any more
      }
      if (lane == 0) wait_fixed(&drain, 0, p.err);
    } else {
      // -------------------------------------------------------------- epilogue warps 2..9
      const int q = warp & 3;              // TMEM lane quarter this warp may access
      const int part = (warp - 2) >> 2;    // this warp takes every other chunk
      constexpr int STEP = 32 * (PG_EPI_WARPS / 4);
      uint8_t* stg = smem + PG_RING + (warp - 2) * PG_STG;
      const uint32_t acce0 = at_leader(smem_u32(acce));
      int ab = 0;
      uint32_t aph = 0;
      EpiRow rr{-1, 0, nullptr};
      int tok = -1, seq = 0, pos = 0;   // the next tile's row, one of its three dependent look-ups at a time
      for (int t = pair; t < total; t += n_pairs) {
        int g, mb, nb;
        locate(t, g, mb, nb);
        const Epi e = p.g[g].epi;
        const int N = p.g[g].N, row0 = rank * 128 + q * 32;
        const int r0 = mb * PG_BM + row0;   // the warp's first row within the group
        const int n_rows = max(0, min(32, s_M[g] - r0));
        int gn = 0;
        if (KIND == EPI_QKV) {
          if (t == pair && lane < n_rows) rr = epi_row(e, s_mbeg[g] + r0 + lane);
          tok = -1;
          if (t + n_pairs < total) {
            int m2, n2;
            locate(t + n_pairs, gn, m2, n2);
            const int r = m2 * PG_BM + row0 + lane;
            if (r < s_M[gn]) tok = p.g[gn].epi.row_tok[s_mbeg[gn] + r];
          }
        }
        const PgTile<KIND> tile{e, stg, lane, s_mbeg[g] + r0, n_rows, nb * BN, min(BN, N - nb * BN), N, pg_vectors<KIND>(e), rr};
        // the first chunk's bias and residual, before the accumulator is there
        typename PgTile<KIND>::In in;
        int c = part * 32;
        tile.load(in, c);
        bool got = true;
        if (lane == 0) got = mbar_wait(&accf[ab], aph, abort_flag, p.err, wlim);
        got = __shfl_sync(0xffffffffu, got ? 1 : 0, 0) != 0;
        if (!got) break;   // warp-uniform: tcgen05.ld below is .sync.aligned
        tc_fence_after();
        const uint32_t tb = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(ab * 256);
        if (KIND == EPI_QKV && tok >= 0) {
          seq = p.g[gn].epi.tok_seq[tok];
          pos = p.g[gn].epi.tok_pos[tok];
        }
#pragma unroll 1
        for (; c < tile.ce; c += STEP) {
          tile.chunk(tb, c, in, acce0 + (uint32_t)ab * 8, c + STEP >= tile.ce);
          tile.load(in, c + STEP);
        }
        if (KIND == EPI_QKV) {
          rr.cbase = tok >= 0 ? p.g[gn].epi.cache.checked_base(p.g[gn].epi.layer0, seq, pos) : -1;
          rr.pos = pos;
        }
        if (part * 32 >= tile.ce && lane == 0) arrive_cluster(acce0 + (uint32_t)ab * 8);   // no chunk of this tile
        ab ^= 1;
        if (ab == 0) aph ^= 1;
      }
    }
  }
  // The pair leaves together. Without a time-out every copy has landed: the MMAs that read it are through (drain).
  __syncthreads();
  if (s_abort) put_peer(smem_u32(&s_stop), rank ^ 1, 1u);   // (by every thread)
  cluster_sync_all();
  if (s_abort || s_stop) pg_leave(full, &s_issued, &s_peer, rank, s_bn, p.err);   // (uniform over the pair)
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
  }
}

// ---------------------------------------------------------------------------- host side
// m-tiles per raster super-row: their A rows (256 x K bf16 each) should take at most ~48 MiB of the 129 MiB L2, leaving
// room for the weight slabs and the output stream.
int pg_raster(int K) { return (int)std::max(1LL, std::min(32LL, (48LL << 20) / std::max(256LL * K * 2, 1LL))); }

template <int KIND, int MAXG>
int pg_pairs() {
  // CTA pairs that are resident at once, 0 when the kernel cannot run
  static int pairs = 0;
  static std::once_flag once;
  std::call_once(once, [] {
    int dev = 0, sms = 0, n = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (cudaFuncSetAttribute(gemm_pair_kernel<KIND, MAXG>, cudaFuncAttributeMaxDynamicSharedMemorySize, PG_SMEM) != cudaSuccess) {
      cudaGetLastError();
      return;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(sms / 2 * 2);
    cfg.blockDim = dim3(PG_THREADS);
    cfg.dynamicSmemBytes = PG_SMEM;
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = 2;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    if (cudaOccupancyMaxActiveClusters(&n, gemm_pair_kernel<KIND, MAXG>, &cfg) != cudaSuccess) {
      cudaGetLastError();
      return;
    }
    pairs = std::min(n, sms / 2);
  });
  return pairs;
}

template <int KIND, int MAXG>
int pg_go(cudaStream_t st, const GemmProblem* probs, int n, unsigned* err) {
  const int pairs = pg_pairs<KIND, MAXG>();
  if (pairs <= 0) return -1;
  thread_local PgParams<MAXG> prm;   // one per host thread
  memset(&prm, 0, sizeof prm);
  prm.n_groups = n;
  prm.err = err;
  for (int i = 0; i < n; ++i) {
    const GemmProblem& q = probs[i];
    PgGroup<MAXG>& g = prm.g[i];
    if (!tc_encode_2d(&g.ta, q.A, (uint64_t)q.K, (uint64_t)q.a_rows, (uint64_t)q.lda * 2, 128)) return -1;
    for (int k = 0; k < PG_N_BN; k += pg_step(MAXG))
      if (!tc_encode_2d(&g.tb[k / pg_step(MAXG)], q.B, (uint64_t)q.K, (uint64_t)q.N, (uint64_t)q.ldb * 2,
                        (uint32_t)(pg_width(k) / 2)))
        return -1;
    g.rows = q.rows;
    g.N = q.N;
    g.K = q.K;
    g.gm = pg_raster(q.K);
    g.epi = q.epi;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(2 * pairs);
  cfg.blockDim = dim3(PG_THREADS);
  cfg.dynamicSmemBytes = PG_SMEM;
  cfg.stream = st;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = 2;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = g_pdl ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, gemm_pair_kernel<KIND, MAXG>, prm) == cudaSuccess ? 1 : -1;
}

}  // namespace

bool pair_gemm_supported(const GemmProblem& q, int max_rows) {
  if (max_rows <= 128 || !tc_gemm_supported()) return false;
  if (q.N <= 0 || q.K <= 0 || q.K % 8 || q.lda % 8 || q.ldb % 8 || q.a_rows <= 0 || q.epi.tile_stats) return false;
  if (((uintptr_t)q.A | (uintptr_t)q.B) & 15) return false;
  // the cache and SwiGLU epilogues work on whole 32-column chunks
  if ((q.epi.kind == EPI_QKV || q.epi.kind == EPI_KV || q.epi.kind == EPI_SWIGLU) && q.N % 32) return false;
  return q.epi.kind >= EPI_F32 && q.epi.kind <= EPI_KV;
}

int pair_gemm(cudaStream_t st, const GemmProblem* probs, int n_probs, const int* max_rows, unsigned* err) {
  if (n_probs < 1 || n_probs > PG_MAXG) return -1;
  // one kernel for EPI_QKV and EPI_KV problems, and one for EPI_F32 and EPI_RESID ones (those without a residual)
  auto kind_of = [](const GemmProblem& q) { return q.epi.kind == EPI_KV ? (int)EPI_QKV : q.epi.kind; };
  int kind = kind_of(probs[0]);
  for (int i = 0; i < n_probs; ++i) {
    if (!pair_gemm_supported(probs[i], max_rows[i])) return -1;
    const int k = kind_of(probs[i]);
    if (k == kind) continue;
    if ((k != EPI_F32 && k != EPI_RESID) || (kind != EPI_F32 && kind != EPI_RESID)) return -1;
    kind = EPI_RESID;
  }
  if (n_probs > 2) {
    switch (kind) {
      case EPI_F32: return pg_go<EPI_F32, PG_MAXG>(st, probs, n_probs, err);
      case EPI_QKV: return pg_go<EPI_QKV, PG_MAXG>(st, probs, n_probs, err);
      default: return -1;
    }
  }
  switch (kind) {
    case EPI_F32: return pg_go<EPI_F32, 2>(st, probs, n_probs, err);
    case EPI_ACT: return pg_go<EPI_ACT, 2>(st, probs, n_probs, err);
    case EPI_RESID: return pg_go<EPI_RESID, 2>(st, probs, n_probs, err);
    case EPI_SWIGLU: return pg_go<EPI_SWIGLU, 2>(st, probs, n_probs, err);
    default: return pg_go<EPI_QKV, 2>(st, probs, n_probs, err);
  }
}

// pg_landing of every stage: out[2 s] what is owed, out[2 s + 1] the parity to wait for.
extern "C" __attribute__((visibility("default"))) void adept_debug_pair_landing(int n0, int n1, int stages, int* out) {
  for (int s = 0; s < stages; ++s) {
    const PgLanding l = pg_landing((uint32_t)n0, (uint32_t)n1, (uint32_t)stages, (uint32_t)s);
    out[2 * s] = (int)l.owe;
    out[2 * s + 1] = (int)l.parity;
  }
}

ADEPT_KTRACE_ATTACH(pg)

ADEPT_WAIT_LIMIT_SETTER(pg)

}  // namespace adept
