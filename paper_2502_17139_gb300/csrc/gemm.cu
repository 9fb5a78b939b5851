// fc_gemm_bf16: C[M][N] = A[M][K] B[K][N] for the decoder forward that
// verifies every draft in one pass (Section IV-D).  Row-major bf16 operands,
// fp32 accumulation in tensor memory, bf16 output.
//
// GB300 design (persistent, warp-specialised tcgen05 kernels, one CTA per SM):
//   * output tiles of 128 x 256; the CTAs walk the tile list with a stride of
//     the grid, M fastest, so the CTAs of a wave share the weight columns they
//     read (and the activations, a few MB, stay in L2);
//   * warp 0 streams 64-deep K slices of A (128 x 64, K-major) and B (64 x 256,
//     N-major: the weights as stored) into a 4-stage ring with TMA (128-byte
//     swizzle; rows and columns past the matrix edge arrive as zeros, so ragged
//     M, N and K need no special case in the main loop);
//   * warp 1 issues tcgen05.mma kind::f16 (M 128, N 256, K 16; four per slice)
//     into one of two tensor-memory accumulators of 256 fp32 columns, and
//     releases each ring stage with a commit when its MMAs are done;
//   * warps 2-5 drain the other accumulator meanwhile (tcgen05.ld, one row per
//     thread), round to bf16 and store the rows; so a tile's epilogue overlaps
//     the next tile's main loop;
//   * every wait is bounded: a wait that runs out raises FC_ERR_TIMEOUT, and
//     the CTA lets its in-flight copies and MMAs land before it frees tensor
//     memory and exits.
//
// The epilogues fold the decoder's next step into the GEMM, so its output
// never makes a round trip through HBM in bf16:
//   * K/V heads (fc_gemm_kv_heads): the fused K/V projection's 256-column
//     tile holds two whole heads (D = 128); the epilogue rotates the key
//     heads by each row's node position (RoPE, rotate-half pairing: columns
//     d and d + 64 of a head, both in the tile) from the fp32 accumulators and
//     writes both kinds head-major, as the tree attention and the cache
//     append read them; fc_gemm_qkv runs the query projection's tiles (stored as
//     they are) and these in one launch;
//   * SiLU * up (fc_gemm_silu_mul): with the gate and up weights interleaved
//     in 128-column blocks (fc_interleave_gate_up), a tile holds gate block t
//     and up block t, and the epilogue writes act[:, 128t .. 128t + 128) =
//     silu(gate) * up.
//
// That is k_gemm, for launches of about one wave of tiles.  k_gemm_pair below
// runs many tiles on pairs of SMs, and k_gemm_split cuts K over the CTAs of a
// cluster where few rows (one user's draft tree is 64 or 128) would leave most
// SMs without a tile.
#include <algorithm>
#include <cmath>
#include <mutex>

#include "fc_common.cuh"

FC_DEFINE_ERROR_WORD(gemm)

namespace {

constexpr int GM_THREADS = 192;  // warp 0 TMA, warp 1 MMA, warps 2-5 epilogue
constexpr int BM = 128, BN = 256, BK = 64, STAGES = 4;
constexpr uint32_t A_BYTES = BM * BK * 2;                // 16 KB
constexpr uint32_t B_CHUNK = BK * 64 * 2;                // 8 KB: 64 K rows x 64 N columns
constexpr uint32_t B_BYTES = (BN / 64) * B_CHUNK;        // 32 KB
constexpr uint32_t STAGE_BYTES = A_BYTES + B_BYTES;      // 48 KB
constexpr uint32_t OFF_BAR = STAGES * STAGE_BYTES;
constexpr uint32_t SMEM_BYTES = OFF_BAR + 256 + 1024;    // + alignment slack
constexpr uint32_t TMEM_COLS = 2 * BN;                   // two accumulators
constexpr uint64_t WAIT_CYCLES = 4000000000ull;          // ~2 s
constexpr uint64_t DRAIN_CYCLES = 400000000ull;          // ~0.2 s

enum { B_FULL = 0, B_EMPTY = STAGES, B_ACC_FULL = 2 * STAGES, B_ACC_EMPTY = 2 * STAGES + 2,
       B_DRAIN = 2 * STAGES + 4, N_BARS = 2 * STAGES + 5 };

enum { EPI_STORE = 0, EPI_KV_HEADS = 1, EPI_SILU_MUL = 2, EPI_QKV = 3 };

struct GemmArgs {
  __nv_bfloat16* c;  // EPI_STORE: C [M][N]; EPI_SILU_MUL: act [M][N / 2]
  int M, N, K;
  int tiles_m, tiles;
  // EPI_KV_HEADS: rows are (sequence, node) = b * n_pad + i; columns are Hkv key
  // heads then Hkv value heads of 128
  __nv_bfloat16* k_out;  // [B][Hkv][n_pad][128], rotated
  __nv_bfloat16* v_out;  // [B][Hkv][n_pad][128]
  const int32_t* pos;    // [B][n_pad]; a negative position leaves its row unrotated
  int n_pad, hkv;
  FcRope64 rope;         // the rotation frequencies
  unsigned int* err;     // the launch's error word (NULL: this file's own)
  int n_q;               // EPI_QKV: columns of the first weights, stored as EPI_STORE does; the rest as EPI_KV_HEADS
};

// The weight map of a column, and the column in it (EPI_QKV has two weight matrices side by side).
template <int EPI>
__device__ __forceinline__ const CUtensorMap* weight_map(const CUtensorMap& b, const CUtensorMap& b2, const GemmArgs& g,
                                                         int& col) {
  if (EPI == EPI_QKV && col >= g.n_q) {
    col -= g.n_q;
    return &b2;
  }
  return &b;
}

__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, int x, int y, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], "
      "[%4];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(bar)
      : "memory");
}

__device__ __forceinline__ void tma_prefetch_2d(const CUtensorMap* map, int x, int y) {
  asm volatile("cp.async.bulk.prefetch.tensor.2d.L2.global.tile [%0, {%1, %2}];" ::"l"(reinterpret_cast<uint64_t>(map)),
               "r"(x), "r"(y)
               : "memory");
}
// Weight slices of a CTA's first tile that k_gemm and k_gemm_pair prefetch while the kernel before drains.  The thread
// that copies issues them, so with nothing to wait for they delay its first copies: us a call, weights from HBM, none /
// 2 / 8: M 4096, K 1024, N 1024 10.5 / 10.6 / 11.4; M 64, K 4096, N 32256 43.7 / 44.2 / 45.8.  Behind a norm they pay,
// two as much as eight (both launches): M 64, K 2048, N 32256 27.7 / 27.1 / 27.4; M 448 51.6 / 50.8 / 50.4.
constexpr int PREFETCH = 2;

__device__ __forceinline__ bool wait_warp(uint32_t bar, uint32_t parity, volatile int* abort) {
  return __all_sync(0xFFFFFFFFu, mbar_wait_bounded(bar, parity, abort, WAIT_CYCLES));
}

__device__ __forceinline__ uint4 pack8_bits(const uint32_t* v) {
  uint4 o;
  o.x = pack_bf16x2(__uint_as_float(v[0]), __uint_as_float(v[1]));
  o.y = pack_bf16x2(__uint_as_float(v[2]), __uint_as_float(v[3]));
  o.z = pack_bf16x2(__uint_as_float(v[4]), __uint_as_float(v[5]));
  o.w = pack_bf16x2(__uint_as_float(v[6]), __uint_as_float(v[7]));
  return o;
}

__device__ __forceinline__ uint4 pack8(const float* v) {
  uint4 o;
  o.x = pack_bf16x2(v[0], v[1]);
  o.y = pack_bf16x2(v[2], v[3]);
  o.z = pack_bf16x2(v[4], v[5]);
  o.w = pack_bf16x2(v[6], v[7]);
  return o;
}

// One output row of a 128 x 256 tile, from 256 tensor-memory columns at tacc
// (one row per thread; called by whole warps).
template <int EPI>
__device__ __forceinline__ void store_tile_row(const GemmArgs& g, uint32_t tacc, int row, int n0, const float2* s_rope,
                                               int ldc = 0) {
  if constexpr (EPI == EPI_QKV) {
    if (n0 < g.n_q) store_tile_row<EPI_STORE>(g, tacc, row, n0, s_rope, g.n_q);
    else store_tile_row<EPI_KV_HEADS>(g, tacc, row, n0 - g.n_q, s_rope);
  } else if constexpr (EPI == EPI_STORE) {
    const int N = ldc ? ldc : g.N;
    __nv_bfloat16* crow = g.c + (size_t)row * N;
#pragma unroll 1
    for (int cc = 0; cc < BN / 32; ++cc) {
      uint32_t v[32];
      tmem_ld32(tacc + cc * 32, v);
      tc_wait_ld();
      const int col = n0 + cc * 32;
      if (row < g.M && col < N) {
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (col + 8 * u + 8 <= N)
            *reinterpret_cast<uint4*>(crow + col + 8 * u) = pack8_bits(v + 8 * u);
      }
    }
  } else if constexpr (EPI == EPI_SILU_MUL) {
    // gate columns [0, 128) and up columns [128, 256) of the tile -> act block n0 / 2
    __nv_bfloat16* arow = g.c + (size_t)row * (g.N / 2) + n0 / 2;
#pragma unroll 1
    for (int cc = 0; cc < 4; ++cc) {
      uint32_t gv[32], uv[32];
      tmem_ld32(tacc + cc * 32, gv);
      tmem_ld32(tacc + 128 + cc * 32, uv);
      tc_wait_ld();
      if (row < g.M) {
        float a[32];
#pragma unroll
        for (int u = 0; u < 32; ++u) {
          const float x = __uint_as_float(gv[u]);
          // the fast divide: an IEEE division takes a slow path for a zero dividend,
          // which doubled this epilogue's time on padding rows (all zeros)
          a[u] = __fdividef(x, 1.f + __expf(-x)) * __uint_as_float(uv[u]);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u)
          *reinterpret_cast<uint4*>(arow + cc * 32 + 8 * u) = pack8(a + 8 * u);
      }
    }
  } else {
    // two heads of 128 columns; head hh < hkv is a key head (rotated)
    const int b = row / g.n_pad, i = row - b * g.n_pad;
    const int p = row < g.M ? g.pos[row] : -1;
#pragma unroll 1
    for (int j = 0; j < 2; ++j) {
      const int hh = n0 / 128 + j;
      const bool key = hh < g.hkv;
      const int head = key ? hh : hh - g.hkv;
      __nv_bfloat16* dst = (key ? g.k_out : g.v_out) + (((size_t)b * g.hkv + head) * g.n_pad + i) * 128;
#pragma unroll 1
      for (int q = 0; q < 2; ++q) {  // dims 32q .. 32q + 31 and their partners 64 + 32q ..
        uint32_t lv[32], hv[32];
        tmem_ld32(tacc + j * 128 + q * 32, lv);
        tmem_ld32(tacc + j * 128 + 64 + q * 32, hv);
        tc_wait_ld();
        if (row < g.M) {
          float lo[32], hi[32];
#pragma unroll
          for (int u = 0; u < 32; ++u) {
            lo[u] = __uint_as_float(lv[u]);
            hi[u] = __uint_as_float(hv[u]);
          }
          if (key && p >= 0) {
#pragma unroll
            for (int u = 0; u < 32; ++u) {
              float sn, cs;
              fc_rope_sincos((float)p, s_rope[q * 32 + u], sn, cs);
              const float x0 = lo[u], x1 = hi[u];
              lo[u] = x0 * cs - x1 * sn;
              hi[u] = x1 * cs + x0 * sn;
            }
          }
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            *reinterpret_cast<uint4*>(dst + q * 32 + 8 * u) = pack8(lo + 8 * u);
            *reinterpret_cast<uint4*>(dst + 64 + q * 32 + 8 * u) = pack8(hi + 8 * u);
          }
        }
      }
    }
  }
}

template <int EPI>
__global__ void __launch_bounds__(GM_THREADS, 1)
    k_gemm(const __grid_constant__ CUtensorMap tm_a, const __grid_constant__ CUtensorMap tm_b,
           const __grid_constant__ CUtensorMap tm_b2, GemmArgs g) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  __shared__ uint32_t s_tmem;
  __shared__ volatile int s_abort;
  __shared__ float2 s_rope[64];
  if constexpr (EPI == EPI_KV_HEADS || EPI == EPI_QKV) fc_rope_copy(s_rope, g.rope);  // read after the barrier below
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  unsigned char* smem =
      reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  const uint32_t sbase = smem_u32(smem);
  const uint32_t bar0 = sbase + OFF_BAR;
  auto bar = [&](int i) { return bar0 + 8u * (uint32_t)i; };
  const int nk = (g.K + BK - 1) / BK;

  if (tid == 0) {
    s_abort = 0;
    for (int i = 0; i < STAGES; ++i) {
      mbar_init(bar(B_FULL + i), 1);
      mbar_init(bar(B_EMPTY + i), 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(bar(B_ACC_FULL + i), 1);
      mbar_init(bar(B_ACC_EMPTY + i), 4);  // one arrival per epilogue warp
    }
    mbar_init(bar(B_DRAIN), 1);
    fence_mbar_init();
    prefetch_tmap(&tm_a);
    prefetch_tmap(&tm_b);
    if constexpr (EPI == EPI_QKV) prefetch_tmap(&tm_b2);
  }
  if (warp == 1) {
    tmem_alloc(smem_u32(&s_tmem), TMEM_COLS);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (tid == 0) {  // the first tile's first weights into L2 while the kernel before drains
    const int n0 = ((int)blockIdx.x / g.tiles_m) * BN;
    for (int kb = 0; kb < min(nk, PREFETCH); ++kb)
      for (int c = 0; c < BN / 64; ++c) {
        int col = n0 + 64 * c;
        const CUtensorMap* m = weight_map<EPI>(tm_b, tm_b2, g, col);
        tma_prefetch_2d(m, col, kb * BK);
      }
  }
  __syncwarp();
  fc_grid_wait();
  const uint32_t tmem = s_tmem;

  if (warp == 0) {
    // ---------------- TMA producer ----------------
    if (lane == 0) {
      uint32_t issued = 0;
      for (int t = blockIdx.x; t < g.tiles && !s_abort; t += gridDim.x) {
        const int m0 = (t % g.tiles_m) * BM;
        int wcol = (t / g.tiles_m) * BN;
        const CUtensorMap* wm = weight_map<EPI>(tm_b, tm_b2, g, wcol);
        for (int kb = 0; kb < nk; ++kb) {
          const uint32_t s = issued % STAGES, ph = (issued / STAGES) & 1;
          if (!mbar_wait_bounded(bar(B_EMPTY + s), ph ^ 1, &s_abort, WAIT_CYCLES)) break;
          const uint32_t st = sbase + s * STAGE_BYTES;
          mbar_expect_tx(bar(B_FULL + s), STAGE_BYTES);
          tma_load_2d(st, &tm_a, kb * BK, m0, bar(B_FULL + s));
#pragma unroll
          for (int c = 0; c < BN / 64; ++c)
            tma_load_2d(st + A_BYTES + c * B_CHUNK, wm, wcol + 64 * c, kb * BK, bar(B_FULL + s));
          ++issued;
        }
      }
      if (s_abort) {  // let the copies in flight land before the CTA exits
        volatile int dummy = 0;
        for (uint32_t i = issued > STAGES ? issued - STAGES : 0; i < issued; ++i)
          mbar_wait_bounded(bar(B_FULL + i % STAGES), (i / STAGES) & 1, &dummy, DRAIN_CYCLES);
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    // ---------------- MMA issuer (the whole warp, one lane elected per MMA) -----
    constexpr uint32_t IDESC = idesc_bf16_f32(BM, BN, 1);  // A K-major, B N-major
    uint32_t consumed = 0, acc_i = 0;
    bool ok = true;
    for (int t = blockIdx.x; ok && t < g.tiles; t += gridDim.x, ++acc_i) {
      const uint32_t buf = acc_i & 1, acc_ph = (acc_i >> 1) & 1;
      if (!(ok = wait_warp(bar(B_ACC_EMPTY + buf), acc_ph ^ 1, &s_abort))) break;
      tc_fence_after();
      const uint32_t d = tmem + buf * BN;
      for (int kb = 0; kb < nk; ++kb, ++consumed) {
        const uint32_t s = consumed % STAGES, ph = (consumed / STAGES) & 1;
        if (!(ok = wait_warp(bar(B_FULL + s), ph, &s_abort))) break;
        tc_fence_after();
        const uint32_t sa = sbase + s * STAGE_BYTES, sb = sa + A_BYTES;
#pragma unroll
        for (int kk = 0; kk < BK / 16; ++kk)
          tc_mma_f16(d, smem_desc_sw128(sa + kk * 32, 16, 1024), smem_desc_sw128(sb + kk * 2048, B_CHUNK, 1024),
                     IDESC, (kb > 0 || kk > 0) ? 1u : 0u);
        tc_commit(bar(B_EMPTY + s));
      }
      if (!ok) break;
      tc_commit(bar(B_ACC_FULL + buf));
    }
    if (__any_sync(0xFFFFFFFFu, s_abort)) {  // let issued MMAs retire before tensor memory is freed
      tc_commit(bar(B_DRAIN));
      volatile int dummy = 0;
      mbar_wait_bounded(bar(B_DRAIN), 0, &dummy, DRAIN_CYCLES);
    }
  } else {
    // ---------------- epilogue: thread = output row of the tile ----------------
    const int q4 = warp & 3;  // the tensor-memory lane quarter this warp may read
    const int r = q4 * 32 + lane;
    const uint32_t lane_off = (uint32_t)(q4 * 32) << 16;
    uint32_t acc_i = 0;
    for (int t = blockIdx.x; t < g.tiles; t += gridDim.x, ++acc_i) {
      const uint32_t buf = acc_i & 1, acc_ph = (acc_i >> 1) & 1;
      if (!wait_warp(bar(B_ACC_FULL + buf), acc_ph, &s_abort)) break;
      tc_fence_after();
      const int m0 = (t % g.tiles_m) * BM, n0 = (t / g.tiles_m) * BN;
      store_tile_row<EPI>(g, tmem + buf * BN + lane_off, m0 + r, n0, s_rope);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar(B_ACC_EMPTY + buf));
    }
  }
  tc_fence_before();
  __syncthreads();
  if (tid == 0 && s_abort) fc_flag(FC_ERR_WORD(g.err), FC_EBIT_TIMEOUT);
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, TMEM_COLS);
  }
}

// ---------------------------------------------------------------------------
// Many tiles: pairs of CTAs (cta_group::2) on tiles of 256 x 256.  A 128 x 256
// tile on one SM moves 12 KB into and 12 KB out of shared memory per 16-deep
// MMA of 128 cycles, 192 bytes a cycle where the SM has 128: k_gemm's tensor
// pipe stands at 68%.  Bound by the MMAs: 1862 TFLOP/s on the LM head (M 2048,
// K 2048, N 32256) where k_gemm reaches 1518.  In a pair each SM holds its own 128 rows of A and half of
// B's columns, 8 KB in and 8 KB out, and the ring is seven slices deep.
//   Both CTAs' copies complete on the leader's (rank 0's) barriers; the leader
// issues the MMAs of both, into tensor memory of both (each its own 128 rows),
// and its commits arrive in both CTAs.  Roles, walk and epilogues as k_gemm.
// ---------------------------------------------------------------------------
constexpr int PR_STAGES = 7, PR_BM = 2 * BM;
constexpr uint32_t PR_B_BYTES = B_BYTES / 2, PR_STAGE = A_BYTES + PR_B_BYTES;  // per CTA: 32 KB
constexpr uint32_t PR_SMEM = PR_STAGES * PR_STAGE + 256 + 1024;                // + barriers + alignment slack
enum { P_FULL = 0, P_EMPTY = PR_STAGES, P_ACC_FULL = 2 * PR_STAGES, P_ACC_EMPTY = P_ACC_FULL + 2,
       P_DRAIN = P_ACC_EMPTY + 2, P_COUNT };
static_assert(P_COUNT * 8 <= 256, "barrier area");

__device__ __forceinline__ uint32_t cluster_addr(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
// A copy into this CTA's shared memory that completes on a barrier of the pair.
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst, const CUtensorMap* map, int x, int y, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], "
      "[%1, {%2, %3}], [%4];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void mma_pair(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                         uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p, e;\n\tsetp.ne.b32 p, %4, 0;\n\telect.sync _|e, 0xffffffff;\n\t"
      "@e tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
      "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// Arrives on the barrier at this offset in both CTAs once the MMAs issued so far are done.
__device__ __forceinline__ void commit_pair(uint32_t bar) {
  asm volatile(
      "{\n\t.reg .pred e;\n\t.reg .b16 m;\n\tmov.b16 m, 3;\n\telect.sync _|e, 0xffffffff;\n\t"
      "@e tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], m;\n\t}" ::"r"(bar)
      : "memory");
}
// An arrival on a barrier of either CTA of the pair (a cluster address).
__device__ __forceinline__ void arrive_cluster(uint32_t addr) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(addr) : "memory");
}
// As mbar_wait_bounded, for a barrier that the other CTA's threads arrive on.
__device__ __forceinline__ bool wait_warp_cluster(uint32_t bar, uint32_t parity, volatile int* abort) {
  const long long t0 = clock64();
  for (;;) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2, 500000;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    if (__all_sync(0xFFFFFFFFu, ok != 0)) return true;
    if (__any_sync(0xFFFFFFFFu, *abort || (uint64_t)(clock64() - t0) > WAIT_CYCLES)) {
      *abort = 1;
      return false;
    }
  }
}

template <int EPI>
__global__ void __launch_bounds__(GM_THREADS, 1) __cluster_dims__(2, 1, 1)
    k_gemm_pair(const __grid_constant__ CUtensorMap tm_a, const __grid_constant__ CUtensorMap tm_b,
           const __grid_constant__ CUtensorMap tm_b2, GemmArgs g) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  __shared__ uint32_t s_tmem;
  __shared__ volatile int s_abort;
  __shared__ float2 s_rope[64];
  if constexpr (EPI == EPI_KV_HEADS || EPI == EPI_QKV) fc_rope_copy(s_rope, g.rope);  // read after the barrier below
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  unsigned char* smem =
      reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  const uint32_t sbase = smem_u32(smem);
  const uint32_t bar0 = sbase + PR_STAGES * PR_STAGE;
  auto bar = [&](int i) { return bar0 + 8u * (uint32_t)i; };
  const int nk = (g.K + BK - 1) / BK;
  const uint32_t rank = cluster_rank();
  const int pair = blockIdx.x >> 1, pairs = gridDim.x >> 1;

  if (tid == 0) {
    s_abort = 0;
    for (int i = 0; i < P_COUNT; ++i)
      mbar_init(bar(i), i == P_ACC_EMPTY || i == P_ACC_EMPTY + 1 ? 8 : 1);  // 4 epilogue warps of both CTAs
    fence_mbar_init();
    prefetch_tmap(&tm_a);
    prefetch_tmap(&tm_b);
    if constexpr (EPI == EPI_QKV) prefetch_tmap(&tm_b2);
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)),
                 "r"(TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();  // both CTAs' barriers are ready
  tc_fence_after();
  if (tid == 0) {  // the first tile's first weights into L2 while the kernel before drains
    const int n0 = (pair / g.tiles_m) * BN + (int)rank * (BN / 2);
    for (int kb = 0; kb < min(nk, PREFETCH); ++kb)
      for (int c = 0; c < BN / 128; ++c) {
        int col = n0 + 64 * c;
        const CUtensorMap* m = weight_map<EPI>(tm_b, tm_b2, g, col);
        tma_prefetch_2d(m, col, kb * BK);
      }
  }
  __syncwarp();
  fc_grid_wait();
  const uint32_t tmem = s_tmem;

  if (warp == 0) {
    // ---------------- TMA producer: this CTA's rows of A, its half of B's columns ----------------
    if (lane == 0) {
      uint32_t issued = 0;
      for (int t = pair; t < g.tiles && !s_abort; t += pairs) {
        const int m0 = (t % g.tiles_m) * PR_BM + (int)rank * BM;
        int wcol = (t / g.tiles_m) * BN + (int)rank * (BN / 2);
        const CUtensorMap* wm = weight_map<EPI>(tm_b, tm_b2, g, wcol);
        for (int kb = 0; kb < nk; ++kb) {
          const uint32_t s = issued % PR_STAGES, ph = (issued / PR_STAGES) & 1;
          if (!mbar_wait_bounded(bar(P_EMPTY + s), ph ^ 1, &s_abort, WAIT_CYCLES)) break;
          const uint32_t st = sbase + s * PR_STAGE, fb = cluster_addr(bar(P_FULL + s), 0);
          if (rank == 0) mbar_expect_tx(bar(P_FULL + s), 2 * PR_STAGE);
          tma_load_2d_pair(st, &tm_a, kb * BK, m0, fb);
#pragma unroll
          for (int c = 0; c < BN / 128; ++c) tma_load_2d_pair(st + A_BYTES + c * B_CHUNK, wm, wcol + 64 * c, kb * BK, fb);
          ++issued;
        }
      }
      if (s_abort && rank == 0) {  // let both CTAs' copies in flight land before either exits
        volatile int dummy = 0;
        for (uint32_t i = issued > PR_STAGES ? issued - PR_STAGES : 0; i < issued; ++i)
          mbar_wait_bounded(bar(P_FULL + i % PR_STAGES), (i / PR_STAGES) & 1, &dummy, DRAIN_CYCLES);
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    // ---------------- MMA issuer: the leader's warp, for both CTAs ----------------
    constexpr uint32_t IDESC = idesc_bf16_f32(PR_BM, BN, 1);  // A K-major, B N-major
    if (rank == 0) {
      uint32_t consumed = 0, acc_i = 0;
      bool ok = true;
      for (int t = pair; ok && t < g.tiles; t += pairs, ++acc_i) {
        const uint32_t buf = acc_i & 1, acc_ph = (acc_i >> 1) & 1;
        if (!(ok = wait_warp_cluster(bar(P_ACC_EMPTY + buf), acc_ph ^ 1, &s_abort))) break;
        tc_fence_after();
        const uint32_t d = tmem + buf * BN;
        for (int kb = 0; kb < nk; ++kb, ++consumed) {
          const uint32_t s = consumed % PR_STAGES, ph = (consumed / PR_STAGES) & 1;
          if (!(ok = wait_warp(bar(P_FULL + s), ph, &s_abort))) break;
          tc_fence_after();
          const uint32_t sa = sbase + s * PR_STAGE, sb = sa + A_BYTES;
#pragma unroll
          for (int kk = 0; kk < BK / 16; ++kk)
            mma_pair(d, smem_desc_sw128(sa + kk * 32, 16, 1024), smem_desc_sw128(sb + kk * 2048, B_CHUNK, 1024), IDESC,
                     (kb > 0 || kk > 0) ? 1u : 0u);
          commit_pair(bar(P_EMPTY + s));
        }
        if (!ok) break;
        commit_pair(bar(P_ACC_FULL + buf));
      }
      if (__any_sync(0xFFFFFFFFu, s_abort)) {  // let issued MMAs retire before tensor memory is freed
        commit_pair(bar(P_DRAIN));
        volatile int dummy = 0;
        mbar_wait_bounded(bar(P_DRAIN), 0, &dummy, DRAIN_CYCLES);
      }
    }
  } else {
    // ---------------- epilogue: thread = output row of this CTA's half of the tile ----------------
    const int q4 = warp & 3;  // the tensor-memory lane quarter this warp may read
    const uint32_t lane_off = (uint32_t)(q4 * 32) << 16;
    uint32_t acc_i = 0;
    for (int t = pair; t < g.tiles; t += pairs, ++acc_i) {
      const uint32_t buf = acc_i & 1, acc_ph = (acc_i >> 1) & 1;
      if (!wait_warp(bar(P_ACC_FULL + buf), acc_ph, &s_abort)) break;
      tc_fence_after();
      const int m0 = (t % g.tiles_m) * PR_BM + (int)rank * BM, n0 = (t / g.tiles_m) * BN;
      store_tile_row<EPI>(g, tmem + buf * BN + lane_off, m0 + q4 * 32 + lane, n0, s_rope);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) arrive_cluster(cluster_addr(bar(P_ACC_EMPTY + buf), 0));
    }
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();  // no CTA leaves while the other's MMAs, copies or arrivals may still reach it
  if (tid == 0 && s_abort) fc_flag(FC_ERR_WORD(g.err), FC_EBIT_TIMEOUT);
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
  }
}

// ---------------------------------------------------------------------------
// Few tiles: the weights are read for so few rows that the work is streaming
// them from HBM, and that needs every SM.  Output tiles of 128 x 64 NB, each
// computed by a cluster of S CTAs that take S consecutive shares of K; a CTA's
// partial tile goes from tensor memory to its shared memory (over its drained
// ring), and after a cluster barrier CTA r sums every S-th group of eight
// columns of both halves over the S partials, in CTA order, and applies the
// epilogue (column c of either half is what the epilogues need together: gate
// and up, or the rotation's partners).  fp32 throughout, no scratch memory.
// Bound by the latency of its steps (a copy, the MMAs, the exchange: 5 us for
// the smallest shape) and then by the weights' stream: the ring is as deep as
// the SM allows (shallower ones, with which the next launch's CTAs would fit
// beside this one's, measured no better).
//   The ring's slices carry only as many rows of A as the matrix has (the MMA
// then reads 128 - a_rows rows of the slice's B as A rows, into accumulator rows
// that nothing reads).
// ---------------------------------------------------------------------------
constexpr int SP_THREADS = 192, SP_MAX_STAGES = 12;
constexpr uint32_t SP_RING_1 = 208 * 1024, SP_RING_2 = 96 * 1024;  // one CTA per SM, or two; a partial tile is 32 NB KB
static_assert(SP_RING_1 >= 4 * 32 * 1024 && SP_RING_2 >= 2 * 32 * 1024, "a partial tile lies in the ring");
constexpr uint32_t SP_EXTRA = 256 + 1024;                       // barriers + alignment slack
enum { SB_FULL = 0, SB_EMPTY = SP_MAX_STAGES, SB_ACC = 2 * SP_MAX_STAGES, SB_DRAIN, SB_COUNT };

struct SplitArgs {
  int a_rows;  // rows of A per slice (a multiple of 8)
  int stages;
  uint32_t ring;  // bytes
};

__device__ __forceinline__ float4 ld_cluster_f4(uint32_t addr, uint32_t rank) {
  float4 v;
  asm volatile(
      "{\n\t.reg .b32 ra;\n\tmapa.shared::cluster.u32 ra, %4, %5;\n\t"
      "ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [ra];\n\t}"
      : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
      : "r"(addr), "r"(rank));
  return v;
}

// Raises the abort flag at this address in all S CTAs of the cluster (before a cluster barrier, so that behind it
// they agree).
template <int S>
__device__ __forceinline__ void abort_cluster(uint32_t flag) {
  for (uint32_t r = 0; r < S; ++r)
    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(cluster_addr(flag, r)), "r"(1u) : "memory");
}

template <int EPI, int S, int NB>
__global__ void __launch_bounds__(SP_THREADS, NB == 2 ? 2 : 1)
    k_gemm_split(const __grid_constant__ CUtensorMap tm_a, const __grid_constant__ CUtensorMap tm_b,
                 const __grid_constant__ CUtensorMap tm_b2, GemmArgs g, SplitArgs sp) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  __shared__ uint32_t s_tmem;
  __shared__ volatile int s_abort;
  __shared__ float2 s_rope[64];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  unsigned char* smem =
      reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  const uint32_t sbase = smem_u32(smem);
  const uint32_t bar0 = sbase + sp.ring;
  auto bar = [&](int i) { return bar0 + 8u * (uint32_t)i; };
  const uint32_t rank = cluster_rank();
  const int t = (int)(blockIdx.x / S), m0 = (t % g.tiles_m) * BM, nt = t / g.tiles_m;
  constexpr int WN = 64 * NB, HN = WN / 2;  // the tile's columns, and those of a half
  // 64-column chunk c of the tile: side by side, but a half of 64 gate columns goes with the same up columns
  auto chunk_col = [&](int c) {
    return EPI == EPI_SILU_MUL && NB == 2 ? 256 * (nt >> 1) + 64 * (nt & 1) + 128 * c : nt * WN + 64 * c;
  };
  const int nk = (g.K + BK - 1) / BK;
  const int k0 = (int)(rank * (uint32_t)nk / S), k1 = (int)((rank + 1) * (uint32_t)nk / S);
  const uint32_t a_bytes = (uint32_t)sp.a_rows * (BK * 2), stage_bytes = a_bytes + NB * B_CHUNK;

  if (tid == 0) {
    s_abort = 0;
    for (int i = 0; i < SB_COUNT; ++i) mbar_init(bar(i), 1);
    fence_mbar_init();
    prefetch_tmap(&tm_a);
    prefetch_tmap(&tm_b);
    if constexpr (EPI == EPI_QKV) prefetch_tmap(&tm_b2);
  }
  if (warp == 1) {
    tmem_alloc(smem_u32(&s_tmem), WN);
    tmem_relinquish();
  }
  if constexpr (EPI == EPI_KV_HEADS || EPI == EPI_QKV) fc_rope_copy(s_rope, g.rope);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  fc_grid_release();
  // this CTA's weights into L2 while the kernel before still runs (a prefetch
  // into the coherent L2 is no read: what that kernel writes to them counts)
  if (tid == 0)
    for (int kb = k0; kb < k1; ++kb)
      for (int c = 0; c < NB; ++c) {
        int col = chunk_col(c);
        const CUtensorMap* m = weight_map<EPI>(tm_b, tm_b2, g, col);
        tma_prefetch_2d(m, col, kb * BK);
      }
  __syncwarp();
  fc_grid_wait();
  const uint32_t tmem = s_tmem;
  const int rows = min(BM, g.M - m0);

  if (warp == 0) {
    if (lane == 0) {  // ---------------- TMA producer ----------------
      int issued = 0;
      for (int kb = k0; kb < k1; ++kb, ++issued) {
        const int s = issued % sp.stages, ph = (issued / sp.stages) & 1;
        if (!mbar_wait_bounded(bar(SB_EMPTY + s), ph ^ 1, &s_abort, WAIT_CYCLES)) break;
        const uint32_t st = sbase + s * stage_bytes, fb = bar(SB_FULL + s);
        mbar_expect_tx(fb, stage_bytes);
#pragma unroll
        for (int c = 0; c < NB; ++c) {
          int col = chunk_col(c);
          const CUtensorMap* m = weight_map<EPI>(tm_b, tm_b2, g, col);
          tma_load_2d(st + a_bytes + c * B_CHUNK, m, col, kb * BK, fb);
        }
        tma_load_2d(st, &tm_a, kb * BK, m0, fb);
      }
      if (s_abort) {  // let the copies in flight land before the CTA exits
        volatile int dummy = 0;
        for (int i = max(0, issued - sp.stages); i < issued; ++i)
          mbar_wait_bounded(bar(SB_FULL + i % sp.stages), (i / sp.stages) & 1, &dummy, DRAIN_CYCLES);
        abort_cluster<S>(smem_u32((const void*)&s_abort));
      }
    }
    __syncwarp();
  } else if (warp == 1) {  // ---------------- MMA issuer ----------------
    constexpr uint32_t IDESC = idesc_bf16_f32(BM, WN, 1);
    bool ok = true;
    for (int i = 0; i < k1 - k0; ++i) {
      const int s = i % sp.stages;
      if (!(ok = wait_warp(bar(SB_FULL + s), (i / sp.stages) & 1, &s_abort))) break;
      tc_fence_after();
      const uint32_t sa = sbase + s * stage_bytes, sb = sa + a_bytes;
#pragma unroll
      for (int kk = 0; kk < BK / 16; ++kk)
        tc_mma_f16(tmem, smem_desc_sw128(sa + kk * 32, 16, 1024), smem_desc_sw128(sb + kk * 2048, B_CHUNK, 1024), IDESC,
                   (i > 0 || kk > 0) ? 1u : 0u);
      tc_commit(bar(SB_EMPTY + s));
    }
    if (ok) tc_commit(bar(SB_ACC));
    if (__any_sync(0xFFFFFFFFu, s_abort)) {  // let issued MMAs retire before tensor memory is freed
      tc_commit(bar(SB_DRAIN));
      volatile int dummy = 0;
      mbar_wait_bounded(bar(SB_DRAIN), 0, &dummy, DRAIN_CYCLES);
      abort_cluster<S>(smem_u32((const void*)&s_abort));
    }
  } else {  // ---------------- warps 2-5: the partial tile to shared memory ----------------
    const int q4 = warp & 3;
    // every MMA has read the ring and every copy has landed: the ring is free
    if (!wait_warp(bar(SB_ACC), 0, &s_abort)) {
      abort_cluster<S>(smem_u32((const void*)&s_abort));
    } else if (q4 * 32 < rows) {
      tc_fence_after();
      float4* red = reinterpret_cast<float4*>(smem) + q4 * 32 + lane;  // [column / 4][row]
#pragma unroll
      for (int cc = 0; cc < WN / 32; ++cc) {
        uint32_t v[32];
        tmem_ld32(tmem + cc * 32 + ((uint32_t)(q4 * 32) << 16), v);
        tc_wait_ld();
#pragma unroll
        for (int u = 0; u < 8; ++u)
          red[(cc * 8 + u) * BM] = make_float4(__uint_as_float(v[4 * u]), __uint_as_float(v[4 * u + 1]),
                                               __uint_as_float(v[4 * u + 2]), __uint_as_float(v[4 * u + 3]));
      }
      tc_fence_before();
    }
  }
  cluster_sync_all();

  // ---------------- this CTA's columns of the tile, eight of each half per item ----------------
  constexpr int QUAD = S < 4 ? S : 4;  // partials whose loads are in flight together
  // groups rank, rank + S, ... of the half's eights; none where a CTA of the cluster gave up: the tile stays as it was
  const int groups = s_abort ? 0 : (HN / 8 - (int)rank + S - 1) / S;
  for (int e = tid; e < rows * groups; e += SP_THREADS) {
    const int cg = e / rows, r = e - cg * rows, c = ((int)rank + cg * S) * 8;
    float lo[8], hi[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) lo[u] = hi[u] = 0.f;
    const uint32_t at = sbase + (uint32_t)((c / 4) * BM + r) * 16;
#pragma unroll
    for (int q0 = 0; q0 < S; q0 += QUAD) {
      float4 v[QUAD][4];
#pragma unroll
      for (int q = 0; q < QUAD; ++q) {
        v[q][0] = ld_cluster_f4(at, q0 + q);
        v[q][1] = ld_cluster_f4(at + BM * 16, q0 + q);
        v[q][2] = ld_cluster_f4(at + (HN / 4) * BM * 16, q0 + q);
        v[q][3] = ld_cluster_f4(at + (HN / 4 + 1) * BM * 16, q0 + q);
      }
#pragma unroll
      for (int q = 0; q < QUAD; ++q) {
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          lo[4 * u] += v[q][u].x, lo[4 * u + 1] += v[q][u].y, lo[4 * u + 2] += v[q][u].z, lo[4 * u + 3] += v[q][u].w;
          hi[4 * u] += v[q][2 + u].x, hi[4 * u + 1] += v[q][2 + u].y;
          hi[4 * u + 2] += v[q][2 + u].z, hi[4 * u + 3] += v[q][2 + u].w;
        }
      }
    }
    const int row = m0 + r;
    const bool plain = EPI == EPI_STORE || (EPI == EPI_QKV && nt * WN < g.n_q);
    if (plain) {
      const int N = EPI == EPI_QKV ? g.n_q : g.N;
      __nv_bfloat16* crow = g.c + (size_t)row * N;
      const int col = nt * WN + c;
      if (col + 8 <= N) *reinterpret_cast<uint4*>(crow + col) = pack8(lo);
      if (col + HN + 8 <= N) *reinterpret_cast<uint4*>(crow + col + HN) = pack8(hi);
    } else if constexpr (EPI == EPI_SILU_MUL) {
#pragma unroll
      for (int u = 0; u < 8; ++u) lo[u] = __fdividef(lo[u], 1.f + __expf(-lo[u])) * hi[u];  // as in k_gemm
      *reinterpret_cast<uint4*>(g.c + (size_t)row * (g.N / 2) + nt * HN + c) = pack8(lo);
    } else if constexpr (EPI != EPI_STORE) {
      const int hh = EPI == EPI_QKV ? nt - g.n_q / 128 : nt;  // the tile is one head
      const int b = row / g.n_pad, i = row - b * g.n_pad;
      const bool key = hh < g.hkv;
      const int head = key ? hh : hh - g.hkv, p = g.pos[row];
      __nv_bfloat16* dst = (key ? g.k_out : g.v_out) + (((size_t)b * g.hkv + head) * g.n_pad + i) * 128 + c;
      if (key && p >= 0) {
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          float sn, cs;
          fc_rope_sincos((float)p, s_rope[c + u], sn, cs);
          const float x0 = lo[u], x1 = hi[u];
          lo[u] = x0 * cs - x1 * sn;
          hi[u] = x1 * cs + x0 * sn;
        }
      }
      *reinterpret_cast<uint4*>(dst) = pack8(lo);
      *reinterpret_cast<uint4*>(dst + 64) = pack8(hi);
    }
  }
  cluster_sync_all();  // no CTA leaves while another may still read its partial tile
  if (tid == 0 && s_abort) fc_flag(FC_ERR_WORD(g.err), FC_EBIT_TIMEOUT);
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, WN);
  }
}

PFN_cuTensorMapEncodeTiled_v12000 get_encode() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  });
  return fn;
}

// Row-major bf16 matrix [rows][cols] as a 2-D map with a (64, box_rows) box,
// 128-byte swizzle; reads past the edges return zeros.
bool make_map_2d(CUtensorMap* m, const void* base, uint64_t rows, uint64_t cols, uint32_t box_rows) {
  auto enc = get_encode();
  if (!enc) return false;
  cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)cols * 2};
  cuuint32_t box[2] = {64, box_rows};
  cuuint32_t es[2] = {1, 1};
  return enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, es,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

int sm_count() {
  int dev = 0, n = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return 0;
  return n;
}

bool aligned16(const void* p) { return reinterpret_cast<uintptr_t>(p) % 16 == 0; }

// How many CTAs a cluster of k_gemm_split has for a launch, 0 = k_gemm.  The
// split kernel serves launches whose 128 x 256 tiles fill less than half of
// the SMs, with the most CTAs that still fit one per SM (a deep ring each);
// shares of K of at least four slices.  The GPCs hold whole clusters: 36 of
// four and 46 of three on 152 SMs, and one more waits for a second wave (M 64,
// K 2048: 47 tiles of three 9.2 -> 15.6 us, 38 of four 8.3 -> 14), hence the
// limits.  Clusters of eight fit two CTAs per SM only (one per SM 10.7 against
// 7.3 us), with half the ring; they pay for up to 64 rows and long K, as those
// of four do there for up to 65 tiles (M 64, K 4096, N 6144: two 16.8, four
// 14.4 us; K 2048: 9.8, 10.0).
// us per call, k_gemm / clusters of 2 / 4 / 8, weights from HBM:
//   M 64,  K 2048, N 2048   13.8 /  9.3 /  7.2 /  7.3      M 512, same        14.7 / 10.7 / 11.5 / 21
//   M 256, K 2048, N 2048   15.1 / 10.3 /  8.4 / 11.1      M 64,  N 4096      14.8 /  9.7 /  8.1 /  8.9
//   M 64,  K 5504, N 2048   31.3 / 17.6 / 11.6 /  9.8      M 128, same        32.6 / 18.7 / 12.6 / 13.3
//   M 512, K 2048, N 4096   15.6 / 14.6 / 23 / 47          (128 big tiles and more: k_gemm)
// Where two CTAs per 128-column tile are too many, clusters of three take
// 256-column tiles: gate/up of inter 5504 at M 64 15.6 -> 12.2, M 128 16.4 -> 14.2.
// Just past clusters of four, those of three: M 64, K 2048, N 5632 9.8 -> 9.0.
struct SplitPlan {
  int cluster, nb;  // CTAs per cluster (0: k_gemm), 64-column chunks per tile
  bool half;        // half the ring, two CTAs per SM
};
SplitPlan choose_split(int M, int64_t tiles_m, int N, int64_t big_tiles, int nk, int sms, bool wide) {
  const int64_t tiles = tiles_m * ((N + 127) / 128);
  if (2 * big_tiles > sms) return {0, 0, false};
  if (M <= 64 && nk >= 64 && tiles * 8 <= sms) return {8, 2, true};
  if (nk >= 16 && tiles * 25 <= 6 * sms) return {4, 2, false};
  if (M <= 64 && nk >= 48 && tiles * 7 <= 3 * sms) return {4, 2, true};
  if (nk >= 12 && tiles * 27 <= 8 * sms) return {3, 2, false};
  if (nk >= 8 && tiles * 2 <= sms) return {2, 2, false};
  return wide && nk >= 12 && big_tiles * 27 <= 8 * sms ? SplitPlan{3, 4, false} : SplitPlan{0, 0, false};
}

// Whether k_gemm_pair serves a launch of `tiles` 128 x 256 tiles: by waves.
// A pair's wave is 3 to 20% shorter at K of 1024 and more, and not below (the
// epilogues are the longer part then), so it may have one wave in eight more,
// which an odd number of row tiles costs it.  One row of tiles would waste
// half of each pair, and in a single wave of short K the pair's set-up (a
// cluster barrier, 0.6 us) is not earned back.  us per call, k_gemm / pairs:
//   M 2048, K 2048, N 32256  178.3 / 145.4    M 2048, K 2048, gate/up 11008  60.2 / 51.2
//   M 2048, K 5504, N 2048    31.6 /  30.1    M 512,  K 2048, N 32256        59.1 / 47.9
//   M 1000, K 2048, N 4096    16.6 /  17.7    M 2048, K 2048, N 2048         15.2 / 15.8
// and with weights from HBM, waves of either in brackets:
//   M 320, K 1024, N 32256 (3, 4)  28.2 / 32.5    M 320, K 4096, N 32256 (3, 4)  84.1 / 84.0
//   M 640, K 4096, gate/up 22016 (3, 4)  78.1 / 81.6
//   M 4096, K 256, N 2048 (2, 2)  9.8 / 11.6      M 3000, K 768, N 8192 (6, 6)  37.6 / 38.4
//   M 4096, K 1024, N 2048 (2, 2)  18.9 / 18.1
bool use_pair(int64_t tiles_m, int64_t tiles, int64_t pair_tiles, int nk, int sms) {
  const int64_t waves = (tiles + sms - 1) / sms, pair_waves = (pair_tiles + sms / 2 - 1) / (sms / 2);
  return tiles_m > 1 && 8 * pair_waves <= 9 * waves && nk >= (waves > 1 ? 16 : 48);
}

template <int EPI>
fc_status launch_gemm(const void* d_a, const void* d_b, int M, int N, int K, GemmArgs g, cudaStream_t stream,
                      const void* d_b2 = nullptr) {
  const int sms = sm_count();
  if (sms <= 0) return FC_ERR_CUDA;
  g.M = M;
  g.N = N;
  g.K = K;
  g.tiles_m = (M + BM - 1) / BM;
  g.err = fc_error_slot();
  const int64_t tiles = (int64_t)g.tiles_m * ((N + BN - 1) / BN);
  if (tiles > 0x7FFFFFFF) return FC_ERR_UNSUPPORTED;
  g.tiles = (int)tiles;
  CUtensorMap ma, mb, mb2;
  constexpr bool WIDE = EPI == EPI_STORE || EPI == EPI_SILU_MUL;  // a narrow tile of the K/V projection is one head
  const SplitPlan plan = choose_split(M, g.tiles_m, N, tiles, (K + BK - 1) / BK, sms, WIDE);
  const int a_rows = plan.cluster ? std::min(BM, (M + 7) / 8 * 8) : BM;
  if (!make_map_2d(&ma, d_a, (uint64_t)M, (uint64_t)K, a_rows) ||
      !make_map_2d(&mb, d_b, (uint64_t)K, (uint64_t)(d_b2 ? g.n_q : N), BK))
    return FC_ERR_CUDA;
  mb2 = mb;
  if (d_b2 && !make_map_2d(&mb2, d_b2, (uint64_t)K, (uint64_t)(N - g.n_q), BK)) return FC_ERR_CUDA;
  using Split = void (*)(CUtensorMap, CUtensorMap, CUtensorMap, GemmArgs, SplitArgs);
  constexpr int W = WIDE ? 4 : 2;
  static constexpr Split narrow[9] = {nullptr, nullptr, k_gemm_split<EPI, 2, 2>, k_gemm_split<EPI, 3, 2>, k_gemm_split<EPI, 4, 2>,
                                      nullptr, nullptr, nullptr, k_gemm_split<EPI, 8, 2>};
  static constexpr Split wide = WIDE ? k_gemm_split<EPI, 3, W> : nullptr;
  static std::atomic<unsigned long long> ready;
  const fc_status set = fc_once_per_device(ready, [](int) -> fc_status {
    if (cudaFuncSetAttribute(k_gemm<EPI>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SMEM_BYTES) != cudaSuccess ||
        cudaFuncSetAttribute(k_gemm_pair<EPI>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)PR_SMEM) != cudaSuccess)
      return FC_ERR_CUDA;
    for (const Split k : {narrow[2], narrow[3], narrow[4], narrow[8], wide})
      if (k && cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(SP_RING_1 + SP_EXTRA)) != cudaSuccess)
        return FC_ERR_CUDA;
    return FC_OK;
  });
  if (set != FC_OK) return set;
  if (plan.cluster) {
    const uint32_t stage = (uint32_t)a_rows * (BK * 2) + plan.nb * B_CHUNK;
    const uint32_t ring = plan.half ? SP_RING_2 : SP_RING_1;
    const SplitArgs sp{a_rows, std::min<int>(SP_MAX_STAGES, ring / stage), ring};
    const int64_t ctas = (int64_t)g.tiles_m * ((N + 64 * plan.nb - 1) / (64 * plan.nb)) * plan.cluster;
    return fc_launch_dependent(plan.nb == 4 ? wide : narrow[plan.cluster], dim3((unsigned)ctas), SP_THREADS,
                               ring + SP_EXTRA, stream, (unsigned)plan.cluster, ma, mb, mb2, g, sp);
  }
  const int64_t pair_tiles = (int64_t)((M + PR_BM - 1) / PR_BM) * ((N + BN - 1) / BN);
  if (use_pair(g.tiles_m, tiles, pair_tiles, (K + BK - 1) / BK, sms)) {
    g.tiles_m = (M + PR_BM - 1) / PR_BM;
    g.tiles = (int)pair_tiles;
    return fc_launch_dependent(k_gemm_pair<EPI>, dim3((unsigned)(2 * std::min(g.tiles, sms / 2))), GM_THREADS, PR_SMEM,
                               stream, 0, ma, mb, mb2, g);
  }
  const int grid = (int)std::min<int64_t>(tiles, sms);
  return fc_launch_dependent(k_gemm<EPI>, dim3((unsigned)grid), GM_THREADS, SMEM_BYTES, stream, 0, ma, mb, mb2, g);
}

// gate/up weights [K][2 * inter] (gate columns, then up columns) -> 128-column
// blocks interleaved: out[:, 256 t + c] = gate[:, 128 t + c] and
// out[:, 256 t + 128 + c] = up[:, 128 t + c], c < 128.  16-byte chunks.
__global__ void k_interleave_gate_up(const uint4* __restrict__ in, uint4* __restrict__ out, int K, int inter) {
  const int cw = inter / 8;  // chunks per half row
  const size_t items = (size_t)K * 2 * cw;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < items; e += (size_t)gridDim.x * blockDim.x) {
    const size_t k = e / (2 * cw);
    const int c = (int)(e - k * 2 * cw);       // output chunk in the row
    const int blk = c / 32, within = c % 32;   // 256-column block, chunk inside it
    const int half = within / 16, cc = within % 16;
    const int src = half * cw + blk * 16 + cc;  // gate or up chunk
    out[e] = in[k * 2 * cw + src];
  }
}

}  // namespace

extern "C" size_t fc_gemm_workspace(void) { return 0; }

extern "C" fc_status fc_gemm_bf16(const void* d_a, const void* d_b, void* d_c, int M, int N, int K, void* d_ws,
                                  size_t ws_bytes, fc_stream stream) {
  FC_NVTX_RANGE();
  (void)d_ws;
  (void)ws_bytes;
  if (M < 0 || N < 1 || K < 1) return FC_ERR_INVALID_ARG;
  if (M == 0) return FC_OK;
  if (!d_a || !d_b || !d_c) return FC_ERR_INVALID_ARG;
  if (!aligned16(d_a) || !aligned16(d_b) || !aligned16(d_c)) return FC_ERR_INVALID_ARG;
  if (N % 8 || K % 8) return FC_ERR_UNSUPPORTED;
  GemmArgs g{};
  g.c = static_cast<__nv_bfloat16*>(d_c);
  return launch_gemm<EPI_STORE>(d_a, d_b, M, N, K, g, static_cast<cudaStream_t>(stream));
}

extern "C" fc_status fc_gemm_kv_heads(const void* d_a, const void* d_wkv, int M, int K, int Hkv, int D, int batch,
                                      int n_pad, const int32_t* d_pos, float rope_base, void* d_k_rot,
                                      void* d_v_heads, fc_stream stream) {
  FC_NVTX_RANGE();
  if (M < 0 || K < 1 || Hkv < 1 || batch < 0 || n_pad < 1 || M != batch * n_pad) return FC_ERR_INVALID_ARG;
  if (D != 128 || K % 8) return FC_ERR_UNSUPPORTED;
  if (!(rope_base > 0.f) || !std::isfinite(rope_base)) return FC_ERR_INVALID_ARG;
  if (M == 0) return FC_OK;
  if (!d_a || !d_wkv || !d_pos || !d_k_rot || !d_v_heads) return FC_ERR_INVALID_ARG;
  if (!aligned16(d_a) || !aligned16(d_wkv) || !aligned16(d_k_rot) || !aligned16(d_v_heads)) return FC_ERR_INVALID_ARG;
  GemmArgs g{};
  g.k_out = static_cast<__nv_bfloat16*>(d_k_rot);
  g.v_out = static_cast<__nv_bfloat16*>(d_v_heads);
  g.pos = d_pos;
  g.n_pad = n_pad;
  g.hkv = Hkv;
  g.rope = fc_rope64(rope_base);
  return launch_gemm<EPI_KV_HEADS>(d_a, d_wkv, M, 2 * Hkv * 128, K, g, static_cast<cudaStream_t>(stream));
}

extern "C" fc_status fc_gemm_qkv(const void* d_a, const void* d_wq, const void* d_wkv, int M, int K, int H, int Hkv, int D,
                                 int batch, int n_pad, const int32_t* d_pos, float rope_base, void* d_q, void* d_k_rot,
                                 void* d_v_heads, fc_stream stream) {
  FC_NVTX_RANGE();
  if (M < 0 || K < 1 || H < 1 || Hkv < 1 || batch < 0 || n_pad < 1 || M != batch * n_pad) return FC_ERR_INVALID_ARG;
  if (D != 128 || K % 8) return FC_ERR_UNSUPPORTED;
  if (!(rope_base > 0.f) || !std::isfinite(rope_base)) return FC_ERR_INVALID_ARG;
  if (M == 0) return FC_OK;
  if (!d_a || !d_wq || !d_wkv || !d_pos || !d_q || !d_k_rot || !d_v_heads) return FC_ERR_INVALID_ARG;
  if (!aligned16(d_a) || !aligned16(d_wq) || !aligned16(d_wkv) || !aligned16(d_q) || !aligned16(d_k_rot) ||
      !aligned16(d_v_heads))
    return FC_ERR_INVALID_ARG;
  if (H % 2) {  // a 256-column tile would hold columns of both
    const fc_status st = fc_gemm_bf16(d_a, d_wq, d_q, M, H * D, K, nullptr, 0, stream);
    return st != FC_OK ? st
                       : fc_gemm_kv_heads(d_a, d_wkv, M, K, Hkv, D, batch, n_pad, d_pos, rope_base, d_k_rot, d_v_heads,
                                          stream);
  }
  GemmArgs g{};
  g.c = static_cast<__nv_bfloat16*>(d_q);
  g.n_q = H * D;
  g.k_out = static_cast<__nv_bfloat16*>(d_k_rot);
  g.v_out = static_cast<__nv_bfloat16*>(d_v_heads);
  g.pos = d_pos;
  g.n_pad = n_pad;
  g.hkv = Hkv;
  g.rope = fc_rope64(rope_base);
  return launch_gemm<EPI_QKV>(d_a, d_wq, M, (H + 2 * Hkv) * D, K, g, static_cast<cudaStream_t>(stream), d_wkv);
}

extern "C" fc_status fc_gemm_silu_mul(const void* d_a, const void* d_wgu, int M, int K, int inter, void* d_act,
                                      fc_stream stream) {
  FC_NVTX_RANGE();
  if (M < 0 || K < 1 || inter < 1) return FC_ERR_INVALID_ARG;
  if (inter % 128 || K % 8) return FC_ERR_UNSUPPORTED;
  if (M == 0) return FC_OK;
  if (!d_a || !d_wgu || !d_act || !aligned16(d_a) || !aligned16(d_wgu) || !aligned16(d_act)) return FC_ERR_INVALID_ARG;
  GemmArgs g{};
  g.c = static_cast<__nv_bfloat16*>(d_act);
  return launch_gemm<EPI_SILU_MUL>(d_a, d_wgu, M, 2 * inter, K, g, static_cast<cudaStream_t>(stream));
}

extern "C" fc_status fc_interleave_gate_up(const void* d_wgu, void* d_out, int K, int inter, fc_stream stream) {
  FC_NVTX_RANGE();
  if (K < 1 || inter < 1) return FC_ERR_INVALID_ARG;
  if (inter % 128) return FC_ERR_UNSUPPORTED;
  if (!d_wgu || !d_out || d_wgu == d_out || !aligned16(d_wgu) || !aligned16(d_out)) return FC_ERR_INVALID_ARG;
  const size_t items = (size_t)K * (2 * inter / 8);
  const unsigned blocks = (unsigned)std::min<size_t>((items + 255) / 256, 152 * 16);
  k_interleave_gate_up<<<blocks, 256, 0, static_cast<cudaStream_t>(stream)>>>(
      static_cast<const uint4*>(d_wgu), static_cast<uint4*>(d_out), K, inter);
  return FC_CHECK_LAUNCH();
}
