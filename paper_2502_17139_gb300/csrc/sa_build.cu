// fc_datastore_build: suffix array + first-token bucket table of a uint32
// token corpus (the datastore organisation of Section IV-A, Eq. 1-2, which
// follows REST's suffix-array index).
//
// Method.  A position's first tokens, as many as fit, are packed into a 64-bit
// key (symbols token + 1, 0 past the corpus end, so a shorter suffix sorts
// first): four tokens at a vocabulary of 32k.  One stable LSD radix sort of
// the keys (8-bit digits, per-block histograms, a global exclusive scan, a
// stable scatter that ranks equal digits inside a warp with __match_any_sync)
// puts every suffix into the range of those that share its key.  Only ranges
// of more than one suffix go on, and each round compares their next tokens:
//   * up to 32 suffixes: a thread per suffix counts those of its range that
//     precede it (k_refine_small, ranges packed into lists);
//   * up to 4096: a CTA sorts the range in shared memory (k_refine_mid);
//   * longer: the ranges' suffixes are gathered and go through the radix sort
//     again, (range, next tokens) as the key.
// Where a range splits, its two neighbours' first different token is their
// common prefix, so the LCP array comes out of the same comparisons.
//
// What the rounds do not resolve ends with prefix doubling over all positions:
// after a round at h every position carries the dense rank of its first h
// tokens (of h or more: ranges that were refined further keep their places),
// and sorting by (rank[i], rank[i + h] + 1) gives the ranks of the first 2h.
// With k tokens a key, that is where
//   * the ranges of more than 4096 suffixes do not halve from one round to the
//     next: a text of more than k or 2k tokens in more than 4096 copies, from
//     h = k on (5M tokens, 5000 copies of 16: 2.6 ms where doubling from the
//     start takes 3.2 and a corpus without them 0.94; 20M, 100000 of 40: 11.6,
//     15.2);
//   * after six rounds a quarter of the suffixes is still in small ranges, or
//     mid ranges have taken n / 2 suffixes through their sort (33 to 4096
//     copies of long texts);
//   * 34 rounds have gone: k tokens each in mid ranges, 8 k to 32 k in small ones
//     (2 to 32 copies of more than about 1000 to 4300 tokens at k = 4).
//
// Bound by HBM: the radix passes stream 32 bytes a position each, the rounds
// gather the text of the suffixes still in play.  Doubling from the start sorts
// all positions in every round: 100M tokens 114 ms against 11.4 ms
// (with the suffix keys); 1M tokens 1.94 against 0.45 ms.

#include <algorithm>

#include "fc_common.cuh"

FC_DEFINE_ERROR_WORD(sa)

namespace {

constexpr int RS_THREADS = 256;
constexpr int RS_ITEMS = 16;
constexpr int RS_TILE = RS_THREADS * RS_ITEMS;  // 4096 keys per block
constexpr int RS_WARPS = RS_THREADS / 32;
constexpr int RS_WARP_CHUNK = 32 * RS_ITEMS;    // 512 consecutive keys per warp

constexpr int SCAN_THREADS = 1024;
constexpr int SCAN_ITEMS = 4;
constexpr int SCAN_TILE = SCAN_THREADS * SCAN_ITEMS;

inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }
inline size_t cdiv(size_t a, size_t b) { return (a + b - 1) / b; }

struct Layout {
  size_t key_a, key_b, val_b, rank, head, hist, scan_tmp, ctl, total;
  size_t nb;          // radix blocks
  size_t scan_len;    // longest array the scan sees
};

size_t scan_tmp_elems(size_t len) {
  size_t t = 0;
  while (len > (size_t)SCAN_TILE) {
    len = cdiv(len, SCAN_TILE);
    t += len;
  }
  return t + 16;
}

Layout layout_for(uint64_t n) {
  Layout L;
  L.nb = cdiv(n, RS_TILE);
  L.scan_len = n > 256 * L.nb ? n : 256 * L.nb;
  size_t off = 0;
  auto take = [&](size_t bytes) {
    size_t o = off;
    off = align_up(off + bytes, 256);
    return o;
  };
  L.key_a = take(n * 8);
  L.key_b = take(n * 8);
  L.val_b = take(n * 4);
  L.rank = take(n * 4);
  L.head = take(n * 4);
  L.hist = take(256 * L.nb * 4);
  L.scan_tmp = take(scan_tmp_elems(L.scan_len) * 4);
  L.ctl = take(64);
  L.total = off;
  return L;
}

// Later rounds: positions in current SA order; key = (rank[i], rank[i+h] + 1 or 0).
// val may alias sa (each element rewrites its own value).
__global__ void k_keys_round(const uint32_t* sa, const uint32_t* __restrict__ rank, uint64_t n, uint64_t h,
                             uint64_t* __restrict__ key, uint32_t* val) {
  for (uint64_t j = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; j < n; j += (uint64_t)gridDim.x * blockDim.x) {
    uint32_t i = sa[j];
    uint64_t lo = ((uint64_t)i + h < n) ? (uint64_t)rank[i + h] + 1 : 0;
    key[j] = ((uint64_t)rank[i] << 32) | lo;
    val[j] = i;
  }
}

struct Sym {
  int bits, count;  // bits per symbol (0..vocab), symbols per key
  uint32_t inv;     // ceil(2^16 / bits): x * inv >> 16 = x / bits for x < 64
};

// The `count` symbols of the suffix at `pos`, the first in the highest bits.
__device__ __forceinline__ uint64_t pack_key(const uint32_t* __restrict__ T, uint64_t n, uint64_t pos, int bits, int count) {
  uint64_t k = 0;
#pragma unroll 4
  for (int j = 0; j < count; ++j) k = (k << bits) | (pos + j < n ? (uint64_t)__ldg(T + pos + j) + 1 : 0ull);
  return k;
}
// The keys of a first pass, made from the text: the positions in order, each with its first symbols.
struct TextKeys {
  const uint32_t* T;
  Sym y;
};

// Per-block histograms of one 8-bit digit.  FIRST: of the text's keys, and the tokens are checked.
template <bool FIRST>
__global__ void __launch_bounds__(RS_THREADS) k_radix_hist(const uint64_t* __restrict__ key, TextKeys tx, uint64_t n, int shift,
                                                           uint32_t* __restrict__ hist, uint64_t nb, uint32_t vocab,
                                                           uint32_t* ctl) {
  __shared__ uint32_t h[256];
  fc_grid_wait();
  key = fc_after_wait(key);
  h[threadIdx.x] = 0;
  __syncthreads();
  const uint64_t base = blockIdx.x * (uint64_t)RS_TILE + threadIdx.x;
  bool bad = false;
  if (FIRST && tx.y.bits < 8) {  // the digit holds several symbols
    for (int k = 0; k < RS_ITEMS; ++k) {
      const uint64_t idx = base + (uint64_t)k * RS_THREADS;
      if (idx >= n) break;
      bad |= __ldg(tx.T + idx) >= vocab;
      atomicAdd(&h[(uint32_t)(pack_key(tx.T, n, idx, tx.y.bits, tx.y.count) >> shift) & 255u], 1u);
    }
  } else {  // every load in flight at once (100M keys 196 us a pass in groups of four loads)
    uint32_t d[RS_ITEMS];  // the digit (FIRST: of the key's last symbol), 256 past the end
#pragma unroll
    for (int k = 0; k < RS_ITEMS; ++k) {
      const uint64_t idx = base + (uint64_t)k * RS_THREADS;
      d[k] = 256u;
      if (idx >= n) continue;
      if constexpr (FIRST) {
        const uint64_t last = idx + (uint64_t)tx.y.count - 1;
        d[k] = last < n ? (__ldg(tx.T + last) + 1u) & 255u : 0u;
        bad |= __ldg(tx.T + idx) >= vocab;
      } else {
        d[k] = (uint32_t)(key[idx] >> shift) & 255u;
      }
    }
#pragma unroll
    for (int k = 0; k < RS_ITEMS; ++k)
      if (d[k] < 256u) atomicAdd(&h[d[k]], 1u);
  }
  if (FIRST && bad) atomicOr(ctl, 1u);
  __syncthreads();
  hist[(uint64_t)threadIdx.x * nb + blockIdx.x] = h[threadIdx.x];
}

// Stable scatter of one 8-bit digit.  offs[d * nb + block] is the exclusive
// scan of the digit-major histogram: where this block's digit-d keys start.
// The block first ranks its keys (per warp with __match_any_sync, then across
// warps and digits), places them in shared memory in digit order, and then
// writes them out in that order: consecutive threads write consecutive
// addresses of a digit's run, so the stores coalesce instead of spraying
// 8- and 4-byte writes over 256 runs.  The values follow through the same
// shared memory.  Bound by the latency of its phases, so by how many blocks an
// SM holds: three at 80 registers (with the values in registers and shared
// memory beside the keys, two: 208 us a pass of 20M pairs against 128).
// FIRST: the keys come from the text and the values are the positions.
template <bool FIRST>
__global__ void __launch_bounds__(RS_THREADS, 3) k_radix_scatter(const uint64_t* __restrict__ kin,
                                                                 const uint32_t* __restrict__ vin, TextKeys tx,
                                                                 uint64_t* __restrict__ kout,
                                                                 uint32_t* __restrict__ vout, uint64_t n, int shift,
                                                                 const uint32_t* __restrict__ offs, uint64_t nb) {
  __shared__ uint64_t skey[RS_TILE];
  uint32_t* sval = reinterpret_cast<uint32_t*>(skey);
  __shared__ uint32_t wbin[RS_WARPS][256];
  __shared__ uint32_t dpos[256];   // where digit d starts in the output, less where it starts in the block's digit order
  __shared__ uint32_t wsum[RS_THREADS / 32];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  for (int d = tid; d < RS_WARPS * 256; d += RS_THREADS) (&wbin[0][0])[d] = 0;
  fc_grid_wait();
  kin = fc_after_wait(kin);
  vin = fc_after_wait(vin);
  offs = fc_after_wait(offs);
  const uint64_t b0 = blockIdx.x * (uint64_t)RS_TILE;
  const uint32_t count = (uint32_t)min((uint64_t)RS_TILE, n - b0);
  const uint64_t w0 = b0 + (uint64_t)warp * RS_WARP_CHUNK + lane;  // this lane's first key; the others every 32
  const int left = (int)count - warp * RS_WARP_CHUNK - lane;       // key `it` exists while 32 it < left
  const uint32_t lt = (1u << lane) - 1u;
  kin += w0;
  vin += w0;
  uint64_t key[RS_ITEMS];
  if constexpr (FIRST) {  // the tile's symbols (0 past the end) and the seven after it, staged
    const int bits = tx.y.bits;
    uint32_t sym[RS_ITEMS + 1];  // every load in flight at once (100M tokens: 1.24 ms one after the other, 0.79 now)
#pragma unroll
    for (int q = 0; q < RS_ITEMS + 1; ++q) {
      const int i = tid + q * RS_THREADS;
      sym[q] = i < RS_TILE + 8 && b0 + i < n ? __ldg(tx.T + b0 + i) + 1u : 0u;
    }
#pragma unroll
    for (int q = 0; q < RS_ITEMS + 1; ++q)
      if (tid + q * RS_THREADS < RS_TILE + 8) sval[tid + q * RS_THREADS] = sym[q];
    __syncthreads();
    const uint32_t* sy = sval + warp * RS_WARP_CHUNK + lane;
    if (tx.y.count == 4 && bits <= 16) {
#pragma unroll
      for (int it = 0; it < RS_ITEMS; ++it)
        key[it] = ((uint64_t)((sy[32 * it] << bits) | sy[32 * it + 1]) << (2 * bits)) |
                  ((sy[32 * it + 2] << bits) | sy[32 * it + 3]);
    } else {
#pragma unroll
      for (int it = 0; it < RS_ITEMS; ++it) {
        uint64_t k = 0;
        for (int j = 0; j < tx.y.count; ++j) k = (k << bits) | sy[32 * it + j];
        key[it] = k;
      }
    }
  } else {
#pragma unroll
    for (int it = 0; it < RS_ITEMS; ++it) key[it] = 32 * it < left ? kin[32 * it] : 0ull;
  }
  const uint32_t base = offs[(uint64_t)tid * nb + blockIdx.x];
  __syncthreads();
  uint32_t at[RS_ITEMS / 2];  // per key, 16 bits: its rank among the warp's equal digits, then its place in the block
#pragma unroll
  for (int it = 0; it < RS_ITEMS; ++it) {
    const bool ok = 32 * it < left;
    const uint32_t d = ok ? ((uint32_t)(key[it] >> shift) & 255u) : 256u;
    const uint32_t peers = __match_any_sync(0xFFFFFFFFu, d);
    // the equal digits' first lane adds them all, behind the iterations before it: other lanes' atomics on a
    // counter are ordered by the warp's barrier alone, and the pass has to be stable
    __syncwarp();
    uint32_t cnt = 0;
    if (ok && (peers & lt) == 0) cnt = atomicAdd(&wbin[warp][d], (uint32_t)__popc(peers));
    const uint32_t r = __shfl_sync(0xFFFFFFFFu, cnt, __ffs(peers) - 1) + __popc(peers & lt);
    at[it / 2] = it & 1 ? at[it / 2] | (r << 16) : r;
  }
  __syncthreads();
  // per digit (thread tid = digit): the digit's block total, then warp prefixes from where it starts in the block
  uint32_t run = 0;
#pragma unroll
  for (int w = 0; w < RS_WARPS; ++w) run += wbin[w][tid];
  uint32_t inc = run;  // exclusive scan of the digit totals over the 256 digits
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, inc, o);
    if (lane >= o) inc += y;
  }
  if (lane == 31) wsum[warp] = inc;
  __syncthreads();
  uint32_t first = inc - run;
  for (int w = 0; w < warp; ++w) first += wsum[w];
  dpos[tid] = base - first;
#pragma unroll
  for (int w = 0; w < RS_WARPS; ++w) {
    const uint32_t c = wbin[w][tid];
    wbin[w][tid] = first;
    first += c;
  }
  __syncthreads();
#pragma unroll
  for (int it = 0; it < RS_ITEMS; ++it) {
    if (32 * it < left) {
      const uint32_t d = (uint32_t)(key[it] >> shift) & 255u;
      const uint32_t p = wbin[warp][d] + ((at[it / 2] >> (16 * (it & 1))) & 0xFFFFu);
      at[it / 2] = it & 1 ? (at[it / 2] & 0xFFFFu) | (p << 16) : (at[it / 2] & 0xFFFF0000u) | p;
      skey[p] = key[it];
    }
  }
  uint32_t val[RS_ITEMS];
#pragma unroll
  for (int it = 0; it < RS_ITEMS; ++it) {
    if constexpr (FIRST) val[it] = (uint32_t)w0 + 32 * it;
    else val[it] = 32 * it < left ? vin[32 * it] : 0u;
  }
  __syncthreads();
  uint32_t pos[RS_ITEMS];
#pragma unroll
  for (int k = 0; k < RS_ITEMS; ++k) {
    const uint32_t j = tid + k * RS_THREADS;
    if (j < count) {
      const uint64_t x = skey[j];
      pos[k] = dpos[(uint32_t)(x >> shift) & 255u] + j;  // positions are below 2^32
      kout[pos[k]] = x;
    }
  }
  __syncthreads();
#pragma unroll
  for (int it = 0; it < RS_ITEMS; ++it)
    if (32 * it < left) sval[(at[it / 2] >> (16 * (it & 1))) & 0xFFFFu] = val[it];
  __syncthreads();
#pragma unroll
  for (int k = 0; k < RS_ITEMS; ++k) {
    const uint32_t j = tid + k * RS_THREADS;
    if (j < count) vout[pos[k]] = sval[j];
  }
}

// All passes over up to RO_MAX pairs in one CTA, the pairs in registers and put
// in order through shared memory: the digits [shift, bits) in steps of eight.
// A pass over a few tiles is three launches that wait for each other (10 us for
// 5000 pairs, six here: a build of 1M tokens 497 -> 468 us).
constexpr int RO_THREADS = 512, RO_WARPS = RO_THREADS / 32, RO_MAX = RO_THREADS * RS_ITEMS;
constexpr uint32_t RO_SMEM = RO_MAX * (8 + 4) + RO_WARPS * 256 * 4;
__global__ void __launch_bounds__(RO_THREADS) k_radix_one(const uint64_t* kin, const uint32_t* vin, uint64_t* kout, uint32_t* vout,
                                                          int m, int shift, int bits) {
  extern __shared__ __align__(16) unsigned char ro_smem[];
  uint64_t* skey = reinterpret_cast<uint64_t*>(ro_smem);
  uint32_t* sval = reinterpret_cast<uint32_t*>(ro_smem + RO_MAX * 8);
  uint32_t* wbin = sval + RO_MAX;  // [warp][256]
  __shared__ uint32_t wsum[8];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int first_item = warp * RS_WARP_CHUNK + lane, left = m - first_item;  // this lane's pairs: every 32
  const uint32_t lt = (1u << lane) - 1u;
  fc_grid_wait();
  uint64_t key[RS_ITEMS];
  uint32_t val[RS_ITEMS], at[RS_ITEMS / 2];
#pragma unroll
  for (int it = 0; it < RS_ITEMS; ++it) {
    key[it] = 32 * it < left ? kin[first_item + 32 * it] : 0ull;
    val[it] = 32 * it < left ? vin[first_item + 32 * it] : 0u;
  }
  for (; shift < bits; shift += 8) {
    for (int d = tid; d < RO_WARPS * 256; d += RO_THREADS) wbin[d] = 0;
    __syncthreads();
#pragma unroll
    for (int it = 0; it < RS_ITEMS; ++it) {
      if (32 * it >= m - warp * RS_WARP_CHUNK) break;  // (the warp has no more)
      const bool ok = 32 * it < left;
      const uint32_t d = ok ? ((uint32_t)(key[it] >> shift) & 255u) : 256u;
      const uint32_t peers = __match_any_sync(0xFFFFFFFFu, d);
      __syncwarp();  // orders the iterations' atomics, as in k_radix_scatter
      uint32_t cnt = 0;
      if (ok && (peers & lt) == 0) cnt = atomicAdd(&wbin[warp * 256 + d], (uint32_t)__popc(peers));
      const uint32_t r = __shfl_sync(0xFFFFFFFFu, cnt, __ffs(peers) - 1) + __popc(peers & lt);
      at[it / 2] = it & 1 ? at[it / 2] | (r << 16) : r;
    }
    __syncthreads();
    uint32_t run = 0, inc = 0;  // threads 0 .. 255: a digit's pairs, and where each warp's start
    if (tid < 256) {
#pragma unroll
      for (int w = 0; w < RO_WARPS; ++w) run += wbin[w * 256 + tid];
      inc = run;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, inc, o);
        if (lane >= o) inc += y;
      }
      if (lane == 31) wsum[warp] = inc;
    }
    __syncthreads();
    if (tid < 256) {
      uint32_t first = inc - run;
      for (int w = 0; w < warp; ++w) first += wsum[w];
#pragma unroll
      for (int w = 0; w < RO_WARPS; ++w) {
        const uint32_t c = wbin[w * 256 + tid];
        wbin[w * 256 + tid] = first;
        first += c;
      }
    }
    __syncthreads();
#pragma unroll
    for (int it = 0; it < RS_ITEMS; ++it) {
      if (32 * it < left) {
        const uint32_t p = wbin[warp * 256 + ((uint32_t)(key[it] >> shift) & 255u)] + ((at[it / 2] >> (16 * (it & 1))) & 0xFFFFu);
        skey[p] = key[it];
        sval[p] = val[it];
      }
    }
    __syncthreads();
#pragma unroll
    for (int it = 0; it < RS_ITEMS; ++it) {
      if (32 * it < left) {
        key[it] = skey[first_item + 32 * it];
        val[it] = sval[first_item + 32 * it];
      }
    }
  }
#pragma unroll
  for (int it = 0; it < RS_ITEMS; ++it) {
    if (32 * it < left) {
      kout[first_item + 32 * it] = key[it];
      vout[first_item + 32 * it] = val[it];
    }
  }
}

// ---- exclusive sum scan of uint32 (three-phase, recursive on the host) ----
__device__ __forceinline__ uint32_t block_exclusive_scan(uint32_t x, uint32_t* total) {
  __shared__ uint32_t warp_sums[SCAN_THREADS / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t inc = x;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    uint32_t y = __shfl_up_sync(0xFFFFFFFFu, inc, o);
    if (lane >= o) inc += y;
  }
  if (lane == 31) warp_sums[warp] = inc;
  __syncthreads();
  if (warp == 0) {
    uint32_t v = (lane < (int)(blockDim.x >> 5)) ? warp_sums[lane] : 0u;
    uint32_t vi = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      uint32_t y = __shfl_up_sync(0xFFFFFFFFu, vi, o);
      if (lane >= o) vi += y;
    }
    warp_sums[lane] = vi - v;
    if (lane == 31) *total = vi;
  }
  __syncthreads();
  uint32_t r = warp_sums[warp] + inc - x;
  __syncthreads();
  return r;
}

__global__ void __launch_bounds__(SCAN_THREADS) k_scan_reduce(const uint32_t* __restrict__ in, uint64_t n,
                                                              uint32_t* __restrict__ partial) {
  __shared__ uint32_t tot;
  fc_grid_wait();
  in = fc_after_wait(in);
  uint64_t base = blockIdx.x * (uint64_t)SCAN_TILE + (uint64_t)threadIdx.x * SCAN_ITEMS;
  uint32_t s = 0;
#pragma unroll
  for (int k = 0; k < SCAN_ITEMS; ++k)
    if (base + k < n) s += in[base + k];
  block_exclusive_scan(s, &tot);
  if (threadIdx.x == 0) partial[blockIdx.x] = tot;
}

__global__ void __launch_bounds__(SCAN_THREADS) k_scan_apply(uint32_t* __restrict__ data, uint64_t n,
                                                             const uint32_t* __restrict__ partial) {
  __shared__ uint32_t tot;
  fc_grid_wait();
  data = fc_after_wait(data);
  partial = fc_after_wait(partial);
  uint64_t base = blockIdx.x * (uint64_t)SCAN_TILE + (uint64_t)threadIdx.x * SCAN_ITEMS;
  uint32_t v[SCAN_ITEMS];
  uint32_t s = 0;
#pragma unroll
  for (int k = 0; k < SCAN_ITEMS; ++k) {
    v[k] = (base + k < n) ? data[base + k] : 0u;
    s += v[k];
  }
  uint32_t pre = block_exclusive_scan(s, &tot) + (partial ? partial[blockIdx.x] : 0u);
#pragma unroll
  for (int k = 0; k < SCAN_ITEMS; ++k) {
    if (base + k < n) data[base + k] = pre;
    pre += v[k];
  }
}

// Up to SC_MAX numbers by one cluster of eight CTAs (the most that is portable),
// each with a stretch of them: one launch instead of three (a build of 1M
// tokens, with eight such scans of 63k: 463 -> 450 us).  Eight numbers a thread
// are two 16-byte loads in flight; the digit counts of 1M tokens just fit, and
// those of more take three launches, each over the whole GPU.
constexpr int SC_CTAS = 8, SC_ITEMS = 8, SC_MAX = SC_CTAS * SCAN_THREADS * SC_ITEMS;
__global__ void __launch_bounds__(SCAN_THREADS) k_scan_cluster(uint32_t* data, uint32_t n) {
  __shared__ uint32_t s_tot;
  fc_grid_wait();
  const uint32_t rank = cluster_rank(), base = (rank * SCAN_THREADS + threadIdx.x) * SC_ITEMS;
  const bool whole = base + SC_ITEMS <= n && reinterpret_cast<uintptr_t>(data) % 16 == 0;
  uint32_t v[SC_ITEMS], sum = 0;
  if (whole) {
#pragma unroll
    for (int k = 0; k < SC_ITEMS; k += 4) {
      const uint4 x = *reinterpret_cast<const uint4*>(data + base + k);
      v[k] = x.x, v[k + 1] = x.y, v[k + 2] = x.z, v[k + 3] = x.w;
    }
  } else {
#pragma unroll
    for (int k = 0; k < SC_ITEMS; ++k) v[k] = base + k < n ? data[base + k] : 0u;
  }
#pragma unroll
  for (int k = 0; k < SC_ITEMS; ++k) sum += v[k];
  uint32_t pre = block_exclusive_scan(sum, &s_tot);
  cluster_sync_all();
  const uint32_t tot = smem_u32(&s_tot);
  for (uint32_t r = 0; r < rank; ++r) {  // the stretches before this one
    uint32_t x;
    asm volatile("{\n\t.reg .b32 ra;\n\tmapa.shared::cluster.u32 ra, %1, %2;\n\tld.shared::cluster.u32 %0, [ra];\n\t}"
                 : "=r"(x)
                 : "r"(tot), "r"(r));
    pre += x;
  }
#pragma unroll
  for (int k = 0; k < SC_ITEMS; ++k) {
    const uint32_t x = v[k];
    v[k] = pre;
    pre += x;
  }
  if (whole) {
#pragma unroll
    for (int k = 0; k < SC_ITEMS; k += 4)
      *reinterpret_cast<uint4*>(data + base + k) = make_uint4(v[k], v[k + 1], v[k + 2], v[k + 3]);
  } else {
#pragma unroll
    for (int k = 0; k < SC_ITEMS; ++k)
      if (base + k < n) data[base + k] = v[k];
  }
  cluster_sync_all();  // no CTA leaves while another may still read its sum
}

cudaError_t exclusive_scan(uint32_t* data, uint64_t n, uint32_t* tmp, cudaStream_t s) {
  if (n == 0) return cudaSuccess;
  if (n > (uint64_t)SCAN_TILE && n <= (uint64_t)SC_MAX)
    return fc_launch_dependent(k_scan_cluster, dim3(SC_CTAS), SCAN_THREADS, 0, s, SC_CTAS, data, (uint32_t)n) == FC_OK
               ? cudaSuccess
               : cudaErrorUnknown;
  uint64_t nt = cdiv(n, SCAN_TILE);
  if (nt > 1) {
    if (fc_launch_dependent(k_scan_reduce, dim3((unsigned)nt), SCAN_THREADS, 0, s, 0, data, n, tmp) != FC_OK)
      return cudaErrorUnknown;
    cudaError_t e = exclusive_scan(tmp, nt, tmp + nt, s);
    if (e != cudaSuccess) return e;
  }
  return fc_launch_dependent(k_scan_apply, dim3((unsigned)nt), SCAN_THREADS, 0, s, 0, data, n,
                             (const uint32_t*)(nt > 1 ? tmp : nullptr)) == FC_OK
             ? cudaSuccess
             : cudaErrorUnknown;
}

// rank[val[j]] = number of distinct keys before position j (dense rank);
// sa[j] = val[j]; ctl[1] = number of distinct keys.
__global__ void k_ranks(const uint64_t* __restrict__ key, const uint32_t* val, const uint32_t* __restrict__ excl,
                        uint64_t n, uint32_t* __restrict__ rank, uint32_t* sa, uint32_t* ctl) {
  for (uint64_t j = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; j < n; j += (uint64_t)gridDim.x * blockDim.x) {
    uint32_t h = (j == 0 || key[j] != key[j - 1]) ? 1u : 0u;
    uint32_t v = val[j];
    rank[v] = excl[j] + h - 1u;
    sa[j] = v;
    if (j == n - 1) ctl[1] = excl[j] + h;
  }
}

__global__ void k_heads(const uint64_t* __restrict__ key, uint64_t n, uint32_t* __restrict__ head) {
  for (uint64_t j = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; j < n; j += (uint64_t)gridDim.x * blockDim.x)
    head[j] = (j == 0 || key[j] != key[j - 1]) ? 1u : 0u;
}

// bucket[v] = first j with T[sa[j]] >= v (binary search), bucket[vocab] = n.
__global__ void k_bucket(const uint32_t* __restrict__ T, const uint32_t* __restrict__ sa, uint64_t n,
                         uint32_t vocab, uint32_t* __restrict__ bucket) {
  for (uint64_t v = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; v <= vocab; v += (uint64_t)gridDim.x * blockDim.x) {
    uint64_t lo = 0, hi = n;
    while (lo < hi) {
      uint64_t mid = (lo + hi) >> 1;
      if (T[sa[mid]] < v) lo = mid + 1;
      else hi = mid;
    }
    bucket[v] = (uint32_t)lo;
  }
}

// lcp[j] = common prefix length of the suffixes at sa[j-1] and sa[j], capped.
// rank is the inverse suffix array; each thread takes one text position i
// (so each suffix is compared with its predecessor in SA order once).
__global__ void k_lcp(const uint32_t* __restrict__ T, const uint32_t* __restrict__ sa,
                      const uint32_t* __restrict__ rank, uint64_t n, uint8_t* __restrict__ lcp) {
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x) {
    const uint32_t j = rank[i];
    uint32_t l = 0;
    if (j > 0) {
      const uint64_t pr = sa[j - 1];
      while (l < FC_LCP_CAP && i + l < n && pr + l < n && T[i + l] == T[pr + l]) ++l;
    }
    lcp[j] = (uint8_t)l;
  }
}

// ---------------------------------------------------------------------------
// Refinement by text (see the top of the file).
// ---------------------------------------------------------------------------
// How many leading symbols two different keys share.
__device__ __forceinline__ uint32_t common_syms(uint64_t a, uint64_t b, const Sym& y) {
  return ((uint32_t)(__clzll((long long)(a ^ b)) - (64 - y.bits * y.count)) * y.inv) >> 16;
}
__device__ __forceinline__ uint8_t cap_lcp(uint32_t l) { return (uint8_t)(l < FC_LCP_CAP ? l : FC_LCP_CAP); }

constexpr uint32_t SMALL_MAX = 32, MID_MAX = 4096;
struct Range {  // a range of suffixes that share their first `depth` tokens
  uint32_t start, size, depth;
};
struct HugeRange {
  uint32_t start, size, depth, base;  // base: its first element among the gathered ones
};
// A list element of a small range: slot (its place in the suffix array) and
// (depth << 8 | its index in the range).
using Elem = uint2;

struct Counts {  // device counters
  uint32_t flag, groups;     // bad token; doubling's number of ranks
  uint32_t small[3], mid[3];  // list elements and ranges: a round reads one, fills the next, clears the third
  uint32_t huge[2], total;
  unsigned long long mid_work;  // suffixes sorted by k_refine_mid so far
};

// Exclusive sum over the block; *total = the whole sum (warps of 32, up to 32 of them).
__device__ __forceinline__ uint32_t block_sum_scan(uint32_t x, uint32_t* wsum, uint32_t* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  uint32_t inc = x;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, inc, o);
    if (lane >= o) inc += y;
  }
  if (lane == 31) wsum[warp] = inc;
  __syncthreads();
  if (warp == 0) {
    const uint32_t v = lane < nw ? wsum[lane] : 0u;
    uint32_t vi = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, vi, o);
      if (lane >= o) vi += y;
    }
    wsum[lane] = vi - v;
    if (lane == 31) *total = vi;
  }
  __syncthreads();
  return wsum[warp] + inc - x;
}

// Splits sorted keys into ranges: the LCP where neighbours differ, the elements
// of small ranges into `small`, longer ranges into `mid` and `huge`.  GATHERED:
// the keys are those of the ranges `from` (their index in the bits above the
// symbols), element a of range r being suffix-array slot start + a - base, and
// `val` is written there; otherwise the keys are all positions', and the
// first-token bucket table is written where `bucket` is given.
constexpr int SPL_THREADS = 256, SPL_TILE = 8 * SPL_THREADS;
template <bool GATHERED>
__global__ void __launch_bounds__(SPL_THREADS) k_split(const uint64_t* __restrict__ key, const uint32_t* __restrict__ val,
                                                       uint64_t m, Sym y, uint32_t depth, const HugeRange* __restrict__ from,
                                                       uint32_t* sa, uint8_t* __restrict__ lcp, Elem* __restrict__ small,
                                                       Range* __restrict__ mid, HugeRange* __restrict__ huge, Counts* ct,
                                                       int huge_out, uint32_t* __restrict__ bucket, uint32_t vocab) {
  __shared__ uint64_t s_key[SPL_TILE + 2 * SMALL_MAX];          // [0]: the key before the tile
  __shared__ uint32_t s_head[SPL_TILE / 32 + 2];               // bit i: element i of the tile starts a range
  __shared__ uint32_t s_list[SPL_TILE / 32 + 1], s_first[SPL_TILE / 32 + 1];  // bit i: it goes to the list; bits before
  __shared__ uint32_t wsum[32], s_total, s_base;
  const int tid = threadIdx.x, lane = tid & 31;
  const uint64_t t0 = blockIdx.x * (uint64_t)SPL_TILE;
  const int have = (int)min((uint64_t)(SPL_TILE + SMALL_MAX), m - t0);  // the tile's elements and the 32 after it
  const int sym_bits = y.bits * y.count;
#pragma unroll
  for (int q = 0; q < SPL_TILE / SPL_THREADS + 1; ++q) {
    const int i = tid + q * SPL_THREADS;
    if (i < have + 1) s_key[i] = (t0 + i > 0) ? key[t0 + i - 1] : ~key[0];  // before the first: any other key
  }
  __syncthreads();
  for (int i = tid; i < SPL_TILE + (int)SMALL_MAX; i += SPL_THREADS) {  // past the end: a range starts
    const uint32_t w = __ballot_sync(0xFFFFFFFFu, i >= have || s_key[i + 1] != s_key[i]);
    if (lane == 0) s_head[i >> 5] = w;
  }
  if (tid == 0) s_head[SPL_TILE / 32 + 1] = 0;  // nothing is known past the 32: such a range is long, or another tile's
  __syncthreads();
  const int tile = min(have, SPL_TILE);
  // an element's slot and the depth that its range now shares
  auto place = [&](int i, uint32_t& slot, uint32_t& d) {
    slot = (uint32_t)(t0 + i);
    d = depth;
    if constexpr (GATHERED) {
      const uint32_t o = (uint32_t)(s_key[i + 1] >> sym_bits);
      slot = from[o].start + (slot - from[o].base);
      d += from[o].depth;
    }
  };
  // an element's range: its head at most 31 back and the next one at most 32 ahead of that, else -1
  auto small_head = [&](int i, bool& alone) -> int {
    const int w = i >> 5, b = i & 31;
    // heads at i - 31 .. i (bit 31 = i) and at i + 1 .. i + 32 (bit 0 = i + 1)
    const uint32_t back = __funnelshift_l(w ? s_head[w - 1] : 0u, s_head[w], 31 - b);
    const uint32_t ahead = __funnelshift_r(b == 31 ? s_head[w + 1] : s_head[w], b == 31 ? 0u : s_head[w + 1], (b + 1) & 31);
    if (!back) return -1;
    const int hd = i - __clz(back);
    const uint32_t to = ahead ? (uint32_t)(i + __ffs(ahead)) : 0xFFFFu;  // the next head
    alone = to - (uint32_t)hd == 1u;
    return hd < tile && to - (uint32_t)hd <= SMALL_MAX ? hd : -1;
  };
  for (int i = tid; i < SPL_TILE + (int)SMALL_MAX; i += SPL_THREADS) {  // whole warps
    bool listed = false;
    if (i < have) {
      bool alone = false;
      const int hd = small_head(i, alone);
      listed = hd >= 0 && !alone;
      if (i < tile) {
        uint32_t slot, d;
        place(i, slot, d);
        if constexpr (GATHERED) sa[slot] = val[t0 + i];
        if ((s_head[i >> 5] >> (i & 31)) & 1u) {
          const uint64_t k = s_key[i + 1], kp = s_key[i];
          if (!GATHERED && bucket) {  // tokens between the neighbours' first ones start here
            const uint32_t ft = (uint32_t)(k >> (sym_bits - y.bits));  // the first token + 1
            for (uint32_t v = t0 + i > 0 ? (uint32_t)(kp >> (sym_bits - y.bits)) : 0u; v < ft; ++v)
              bucket[v] = (uint32_t)(t0 + i);
          }
          if (GATHERED ? (t0 + i > 0 && (kp >> sym_bits) == (k >> sym_bits)) : t0 + i > 0)
            lcp[slot] = cap_lcp(d - (uint32_t)y.count + common_syms(k, kp, y));
          else if (!GATHERED)
            lcp[slot] = 0;
          if (hd < 0) {  // a longer range: its end by doubling steps and bisection over the sorted keys
            uint64_t lo = t0 + i + SMALL_MAX, step = SMALL_MAX;  // key[lo - 1] belongs to it
            while (lo - 1 + step < m && key[lo - 1 + step] == k) {
              lo += step;
              step *= 2;
            }
            uint64_t hi = min(m, lo - 1 + step);  // the first element past it lies in [lo, hi]
            while (lo < hi) {
              const uint64_t c = (lo + hi) >> 1;
              if (key[c] == k) lo = c + 1;
              else hi = c;
            }
            const uint32_t size = (uint32_t)(lo - (t0 + i));
            if (size <= MID_MAX) mid[atomicAdd(&ct->mid[0], 1u)] = Range{slot, size, d};
            else huge[atomicAdd(&ct->huge[huge_out], 1u)] = HugeRange{slot, size, d, 0u};
          }
        }
      }
    }
    const uint32_t w = __ballot_sync(0xFFFFFFFFu, listed);
    if (lane == 0) s_list[i >> 5] = w;
  }
  if (!GATHERED && bucket && t0 + tile == m)  // and none after the last suffix's
    for (uint32_t v = (uint32_t)(s_key[tile] >> (sym_bits - y.bits)) + tid; v <= vocab; v += SPL_THREADS) bucket[v] = (uint32_t)m;
  __syncthreads();
  const uint32_t cnt = tid < SPL_TILE / 32 + 1 ? (uint32_t)__popc(s_list[tid]) : 0u;
  const uint32_t first = block_sum_scan(cnt, wsum, &s_total);
  if (tid < SPL_TILE / 32 + 1) s_first[tid] = first;
  if (tid == 0 && s_total) s_base = atomicAdd(&ct->small[0], s_total);
  __syncthreads();
  for (int i = tid; i < SPL_TILE + (int)SMALL_MAX; i += SPL_THREADS) {
    const uint32_t w = s_list[i >> 5];
    if (!((w >> (i & 31)) & 1u)) continue;
    uint32_t slot, d;
    bool alone;
    place(i, slot, d);
    small[s_base + s_first[i >> 5] + __popc(w & ((1u << (i & 31)) - 1u))] =
        make_uint2(slot, (d << 8) | (uint32_t)(i - small_head(i, alone)));
  }
}

// One round over the small ranges: a tile of 256 list elements holds the whole
// of every range that starts in its first 224.  A thread compares its suffix's
// next symbols with those of its range: how many are smaller (its new
// sub-range's place), equal (they go on), and the largest smaller one (the LCP
// at the new sub-range's start).  Several rounds run in the tile before what is
// left goes back to a list: the next symbols lie beside the last ones, and a
// launch and a list's way through memory are saved (a build of 1M tokens
// 628 -> 533 us, of 100M 13.3 -> 12.9 ms).  Where every tile has its own CTA there is
// nothing to gain from packing: RFS_DEEP rounds.  Else `many`: one in the first
// round, which leaves a quarter of its elements, then eight (an eighth goes
// each round).
constexpr int RFS_DEEP = 32;
constexpr int RFS_THREADS = 256, RFS_HEADS = RFS_THREADS - (int)SMALL_MAX;
__global__ void __launch_bounds__(RFS_THREADS) k_refine_small(const uint32_t* __restrict__ T, uint64_t n, Sym y, uint32_t* sa,
                                                              uint8_t* __restrict__ lcp, const Elem* list, Elem* next,
                                                              Counts* ct, int in, int out, int many) {
  __shared__ uint64_t s_key[RFS_THREADS];
  __shared__ uint32_t s_idx[RFS_THREADS + 1], s_act[RFS_THREADS], s_pos[RFS_THREADS], wsum[32], s_total, s_base;
  __shared__ Elem s_out[RFS_THREADS];
  const int tid = threadIdx.x;
  fc_grid_wait();
  const uint32_t m = *(volatile uint32_t*)&ct->small[in];
  const uint32_t tiles = m / RFS_HEADS + (m % RFS_HEADS != 0);
  const int deep = tiles <= gridDim.x ? RFS_DEEP : many;
  for (uint32_t t = blockIdx.x; t < tiles; t += gridDim.x) {
    const uint64_t a = (uint64_t)t * RFS_HEADS + tid;
    Elem e = a < m ? list[a] : make_uint2(0u, 0u);
    uint32_t idx = e.y & 255u, d = e.y >> 8;
    int hd = tid - (int)idx;  // the range's first element in the tile
    bool mine = a < m && hd >= 0 && hd < RFS_HEADS;
    uint32_t pos = mine ? sa[e.x] : 0u, act;
    for (int r = 1;; ++r) {
      const uint64_t k = mine ? pack_key(T, n, (uint64_t)pos + d, y.bits, y.count) : 0ull;
      s_key[tid] = k;
      s_idx[tid] = mine || r == 1 ? idx : 0u;
      if (tid == 0) s_idx[RFS_THREADS] = 0u;
      s_act[tid] = 0u;
      __syncthreads();
      if (mine) {
        uint32_t less = 0, before = 0, equal = 0;
        uint64_t below = 0;
        for (int j = hd; j == hd || s_idx[j] != 0u; ++j) {  // the next range (or the end) starts at index 0
          const uint64_t o = s_key[j];
          if (o < k) {
            ++less;
            below = max(below, o);
          } else if (o == k) {
            ++equal;
            before += j < tid;
          }
        }
        const uint32_t slot = e.x - idx + less + before;
        sa[slot] = pos;
        if (before == 0 && less > 0) lcp[slot] = cap_lcp(d + common_syms(k, below, y));
        if (equal > 1) {
          const int at = hd + (int)(less + before);
          s_act[at] = 1u;
          s_pos[at] = pos;
          s_out[at] = make_uint2(slot, ((d + (uint32_t)y.count) << 8) | before);
        }
      }
      __syncthreads();
      act = s_act[tid];
      if (r >= deep || !__syncthreads_or((int)act)) break;
      mine = act != 0;
      if (mine) e = s_out[tid];
      pos = s_pos[tid];
      idx = e.y & 255u;
      d = e.y >> 8;
      hd = tid - (int)idx;
    }
    const uint32_t at = block_sum_scan(act, wsum, &s_total);
    if (tid == 0 && s_total) s_base = atomicAdd(&ct->small[out], s_total);
    __syncthreads();
    if (act) next[s_base + at] = s_out[tid];
    __syncthreads();
  }
}

// One round over the ranges of 33 to 4096 suffixes: a group of threads sorts a
// range's (next symbols, position) pairs in shared memory (bitonic) and splits
// it.  Bound by the latency of the sort's steps, so by how many ranges an SM has
// in work: 64 threads take a range of up to 512, the whole CTA a longer one
// (100M tokens: 1097 us a round with a CTA for each, 605 now).
constexpr int RFM_THREADS = 512, RFM_GROUP = 64, RFM_GROUPS = RFM_THREADS / RFM_GROUP;
constexpr uint32_t RFM_GROUP_MAX = MID_MAX / RFM_GROUPS, RFM_SMEM = MID_MAX * (8 + 4);
struct MidShared {  // one range's: key and position arrays for its size, heads, and a few words
  uint64_t* key;
  uint32_t *pos, *head, *wsum, *base;
};
template <int NT>
__device__ __forceinline__ void mid_sync(int bar) {
  asm volatile("bar.sync %0, %1;" ::"r"(bar), "n"(NT) : "memory");
}
// One range by NT threads (tid: within them), whose barrier is `bar`.
template <int NT>
__device__ __forceinline__ void mid_range(const Range g, const MidShared sh, int tid, int bar, const uint32_t* __restrict__ T,
                                          uint64_t n, Sym y, uint32_t* sa, uint8_t* __restrict__ lcp, Range* next, Elem* small,
                                          Counts* ct, int out) {
  const int lane = tid & 31, warp = tid >> 5;
  if (tid == 0) atomicAdd(&ct->mid_work, (unsigned long long)g.size);
  uint32_t p2 = 64;
  while (p2 < g.size) p2 *= 2;
  for (uint32_t i = tid; i < p2; i += NT) {
    uint32_t pos = 0xFFFFFFFFu;  // padding sorts behind every suffix
    uint64_t k = ~0ull;
    if (i < g.size) {
      pos = sa[g.start + i];
      k = pack_key(T, n, (uint64_t)pos + g.depth, y.bits, y.count);
    }
    sh.key[i] = k;
    sh.pos[i] = pos;
  }
  mid_sync<NT>(bar);
  for (uint32_t len = 2; len <= p2; len *= 2)
    for (uint32_t st = len / 2; st > 0; st /= 2) {
      for (uint32_t i = tid; i < p2 / 2; i += NT) {
        const uint32_t a = 2 * i - (i & (st - 1)), b = a + st;
        const uint64_t ka = sh.key[a], kb = sh.key[b];
        const uint32_t pa = sh.pos[a], pb = sh.pos[b];
        const bool up = (a & len) == 0, gt = ka > kb || (ka == kb && pa > pb);
        if (gt == up) {
          sh.key[a] = kb, sh.key[b] = ka;
          sh.pos[a] = pb, sh.pos[b] = pa;
        }
      }
      // a step of up to 32 stays in its warp's 64 elements
      if (st >= 64 || (st == 1 && len >= 64)) mid_sync<NT>(bar);  // (the next step's is st / 2, or len)
      else __syncwarp();
    }
  const uint32_t words = (g.size + 31) / 32 + 1;
  for (uint32_t i = tid; i < words * 32; i += NT) {
    const bool head = i >= g.size || i == 0 || sh.key[i] != sh.key[i - 1];
    const uint32_t w = __ballot_sync(0xFFFFFFFFu, head);  // whole warps: words * 32 elements
    if (lane == 0) sh.head[i >> 5] = w;
  }
  mid_sync<NT>(bar);
  // a thread takes consecutive elements, so that its small ones stay in order
  const uint32_t per = (g.size + NT - 1) / NT, i0 = min(g.size, tid * per), i1 = min(g.size, i0 + per);
  auto range_of = [&](uint32_t i, uint32_t& hd, uint32_t& nx) {  // the bounds of i's sub-range
    uint32_t w = i >> 5, v = sh.head[w] & (0xFFFFFFFFu >> (31 - (i & 31)));
    while (!v) v = sh.head[--w];  // element 0 is a head
    hd = w * 32 + 31 - __clz(v);
    w = (i + 1) >> 5, v = sh.head[w] & (0xFFFFFFFFu << ((i + 1) & 31));
    while (!v) v = sh.head[++w];  // the word past the last element is all heads
    nx = min(g.size, w * 32 + __ffs(v) - 1);
  };
  uint32_t n_out = 0;
  for (uint32_t i = i0; i < i1; ++i) {
    sa[g.start + i] = sh.pos[i];
    uint32_t hd, nx;
    range_of(i, hd, nx);
    const uint32_t size = nx - hd;
    if (i == hd && i > 0) lcp[g.start + i] = cap_lcp(g.depth + common_syms(sh.key[i], sh.key[i - 1], y));
    if (size > SMALL_MAX) {
      if (i == hd) next[atomicAdd(&ct->mid[out], 1u)] = Range{g.start + hd, size, g.depth + (uint32_t)y.count};
    } else if (size > 1) {
      ++n_out;
    }
  }
  uint32_t inc = n_out;  // the small ones before this thread's
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t v = __shfl_up_sync(0xFFFFFFFFu, inc, o);
    if (lane >= o) inc += v;
  }
  if (lane == 31) sh.wsum[warp] = inc;
  mid_sync<NT>(bar);
  uint32_t at = inc - n_out, total = 0;
#pragma unroll
  for (int w = 0; w < NT / 32; ++w) {
    const uint32_t v = sh.wsum[w];
    at += w < warp ? v : 0u;
    total += v;
  }
  if (tid == 0 && total) *sh.base = atomicAdd(&ct->small[out], total);
  mid_sync<NT>(bar);
  at += *sh.base;
  if (n_out)
    for (uint32_t i = i0; i < i1; ++i) {
      uint32_t hd, nx;
      range_of(i, hd, nx);
      if (nx - hd > 1 && nx - hd <= SMALL_MAX)
        small[at++] = make_uint2(g.start + i, ((g.depth + (uint32_t)y.count) << 8) | (i - hd));
    }
  mid_sync<NT>(bar);
}
__global__ void __launch_bounds__(RFM_THREADS) k_refine_mid(const uint32_t* __restrict__ T, uint64_t n, Sym y, uint32_t* sa,
                                                            uint8_t* __restrict__ lcp, const Range* ranges, Range* next,
                                                            Elem* small, Counts* ct, int in, int out) {
  extern __shared__ __align__(16) unsigned char rfm_smem[];
  __shared__ uint32_t s_head[MID_MAX / 32 + 2 * RFM_GROUPS], s_wsum[RFM_THREADS / 32], s_base[RFM_GROUPS];
  const int tid = threadIdx.x, lane = tid & 31, grp = tid / RFM_GROUP;
  fc_grid_wait();
  const uint32_t ng = *(volatile uint32_t*)&ct->mid[in];
  if (blockIdx.x == 0 && tid == 0) ct->small[3 - in - out] = ct->mid[3 - in - out] = 0u;  // the round after next's
  uint64_t* key = reinterpret_cast<uint64_t*>(rfm_smem);
  uint32_t* pos = reinterpret_cast<uint32_t*>(rfm_smem + MID_MAX * 8);
  const MidShared part{key + grp * RFM_GROUP_MAX, pos + grp * RFM_GROUP_MAX, s_head + grp * (RFM_GROUP_MAX / 32 + 2),
                       s_wsum + grp * (RFM_GROUP / 32), s_base + grp};
  for (uint32_t gi = blockIdx.x * RFM_GROUPS + grp; gi < ng; gi += gridDim.x * RFM_GROUPS) {
    const Range g = ranges[gi];
    if (g.size <= RFM_GROUP_MAX)
      mid_range<RFM_GROUP>(g, part, tid % RFM_GROUP, 1 + grp, T, n, y, sa, lcp, next, small, ct, out);
  }
  __syncthreads();
  const MidShared all{key, pos, s_head, s_wsum, s_base};
  for (uint32_t g0 = blockIdx.x; g0 < ng; g0 += gridDim.x * 32) {  // 32 of this CTA's ranges at a time
    const uint32_t mine = g0 + lane * gridDim.x;
    uint32_t longer = __ballot_sync(0xFFFFFFFFu, mine < ng && ranges[mine].size > RFM_GROUP_MAX);
    for (; longer; longer &= longer - 1)
      mid_range<RFM_THREADS>(ranges[g0 + (__ffs(longer) - 1) * gridDim.x], all, tid, 1 + RFM_GROUPS, T, n, y, sa, lcp, next,
                             small, ct, out);
  }
}

// base[] of the huge ranges (one CTA) and their total.
__global__ void __launch_bounds__(SCAN_THREADS) k_huge_base(HugeRange* r, Counts* ct, int in) {
  __shared__ uint32_t tot;
  const uint32_t ng = ct->huge[in];
  uint32_t run = 0;
  for (uint32_t t = 0; t < ng; t += SCAN_THREADS) {
    const uint32_t i = t + threadIdx.x, s = i < ng ? r[i].size : 0u;
    const uint32_t ex = block_exclusive_scan(s, &tot);
    if (i < ng) r[i].base = run + ex;
    run += tot;
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    ct->total = run;
    ct->huge[in ^ 1] = 0;
  }
}

// The huge ranges' suffixes with (range, next symbols) keys.
__global__ void k_huge_gather(const uint32_t* __restrict__ T, uint64_t n, Sym y, const uint32_t* __restrict__ sa,
                              const HugeRange* __restrict__ r, uint32_t ng, uint32_t m, uint64_t* __restrict__ key,
                              uint32_t* __restrict__ val) {
  for (uint64_t a = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; a < m; a += (uint64_t)gridDim.x * blockDim.x) {
    uint32_t lo = 0, hi = ng;  // the last range with base <= a
    while (hi - lo > 1) {
      const uint32_t c = (lo + hi) >> 1;
      if (r[c].base <= a) lo = c;
      else hi = c;
    }
    const uint32_t pos = sa[r[lo].start + ((uint32_t)a - r[lo].base)];
    key[a] = ((uint64_t)lo << (y.bits * y.count)) | pack_key(T, n, (uint64_t)pos + r[lo].depth, y.bits, y.count);
    val[a] = pos;
  }
}

// Where prefix doubling takes over: every position's rank is the first slot of its range.
__global__ void k_rank_slots(const uint32_t* __restrict__ sa, uint64_t n, uint32_t* __restrict__ rank) {
  for (uint64_t j = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; j < n; j += (uint64_t)gridDim.x * blockDim.x)
    rank[sa[j]] = (uint32_t)j;
}
__global__ void k_rank_ranges(const uint32_t* __restrict__ sa, const Elem* __restrict__ list, const Range* __restrict__ mid,
                              const HugeRange* __restrict__ huge, const Counts* ct, int in, int huge_in,
                              uint32_t* __restrict__ rank) {
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x, t = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
  for (uint64_t a = t; a < ct->small[in]; a += stride) rank[sa[list[a].x]] = list[a].x - (list[a].y & 255u);
  for (uint32_t g = blockIdx.x; g < ct->mid[in]; g += gridDim.x)
    for (uint32_t i = threadIdx.x; i < mid[g].size; i += blockDim.x) rank[sa[mid[g].start + i]] = mid[g].start;
  for (uint32_t g = 0; g < ct->huge[huge_in]; ++g)
    for (uint64_t i = t; i < huge[g].size; i += stride) rank[sa[huge[g].start + i]] = huge[g].start;
}

int sm_count() {
  int dev = 0, n = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return 0;
  return n;
}

inline int bits_for(uint64_t x) {
  int b = 0;
  while (x) {
    ++b;
    x >>= 1;
  }
  return b;
}

inline unsigned grid_for(uint64_t n, int threads) {
  uint64_t g = cdiv(n, threads);
  if (g > 152ull * 64) g = 152ull * 64;
  return (unsigned)(g ? g : 1);
}

}  // namespace

extern "C" size_t fc_datastore_build_workspace(uint64_t n_tokens, uint32_t vocab) {
  (void)vocab;
  if (n_tokens == 0) return 0;
  return layout_for(n_tokens).total;
}

extern "C" fc_status fc_datastore_build(const uint32_t* d_tokens, uint64_t n, uint32_t vocab, uint32_t* d_sa,
                                        uint32_t* d_bucket, uint8_t* d_lcp, void* d_ws, size_t ws_bytes,
                                        fc_stream stream, fc_datastore* out) {
  FC_NVTX_RANGE();
  if (!d_tokens || !d_sa || !d_bucket || !d_lcp || n == 0 || n >= 0xFFFFFFFFull || vocab == 0 ||
      vocab >= 0x80000000u)
    return FC_ERR_INVALID_ARG;
  Layout L = layout_for(n);
  if (!d_ws || ws_bytes < L.total) return FC_ERR_WORKSPACE;
  if (reinterpret_cast<uintptr_t>(d_ws) % 256) return FC_ERR_INVALID_ARG;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  char* ws = static_cast<char*>(d_ws);
  uint64_t* key_a = reinterpret_cast<uint64_t*>(ws + L.key_a);
  uint64_t* key_b = reinterpret_cast<uint64_t*>(ws + L.key_b);
  uint32_t* val_b = reinterpret_cast<uint32_t*>(ws + L.val_b);
  uint32_t* rank = reinterpret_cast<uint32_t*>(ws + L.rank);
  uint32_t* head = reinterpret_cast<uint32_t*>(ws + L.head);
  uint32_t* hist = reinterpret_cast<uint32_t*>(ws + L.hist);
  uint32_t* stmp = reinterpret_cast<uint32_t*>(ws + L.scan_tmp);
  uint32_t* ctl = reinterpret_cast<uint32_t*>(ws + L.ctl);
  const unsigned g = grid_for(n, 256);
  Counts* ct = reinterpret_cast<Counts*>(ctl);
  Counts hc{};
  static_assert(sizeof(Counts) <= 64, "counter area");
  auto read_counts = [&]() -> bool {  // synchronises
    return cudaMemcpyAsync(&hc, ct, sizeof hc, cudaMemcpyDeviceToHost, s) == cudaSuccess &&
           cudaStreamSynchronize(s) == cudaSuccess;
  };
  // One pass of an LSD sort of m (key, value) pairs: digit offsets, then the scatter.
  auto offsets = [&](uint64_t m) { return exclusive_scan(hist, 256 * cdiv(m, RS_TILE), stmp, s) == cudaSuccess; };
  auto pass = [&](const uint64_t* kin, const uint32_t* vin, uint64_t* kout, uint32_t* vout, uint64_t m, int shift) {
    const uint64_t nb = cdiv(m, RS_TILE);
    return fc_launch_dependent(k_radix_hist<false>, dim3((unsigned)nb), RS_THREADS, 0, s, 0, kin, TextKeys{}, m, shift, hist, nb,
                               0u, nullptr) == FC_OK &&
           offsets(m) &&
           fc_launch_dependent(k_radix_scatter<false>, dim3((unsigned)nb), RS_THREADS, 0, s, 0, kin, vin, TextKeys{}, kout, vout,
                               m, shift, hist, nb) == FC_OK;
  };
  // The passes from digit `d` on over the low `bits` bits, from one pair of buffers to the other.
  auto passes = [&](uint64_t* k0, uint32_t* v0, uint64_t* k1, uint32_t* v1, uint64_t m, int d, int bits) {
    if (m <= (uint64_t)RO_MAX && 8 * d < bits) {
      const bool odd = ((bits - 8 * d + 7) / 8) % 2 != 0;
      return fc_launch_dependent(k_radix_one, dim3(1), RO_THREADS, RO_SMEM, s, 0, k0, v0, odd ? k1 : k0, odd ? v1 : v0, (int)m,
                                 8 * d, bits) == FC_OK;
    }
    for (; 8 * d < bits; ++d) {
      if (!pass(k0, v0, k1, v1, m, 8 * d)) return false;
      std::swap(k0, k1);
      std::swap(v0, v1);
    }
    return true;
  };

  if (cudaFuncSetAttribute(k_refine_mid, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)RFM_SMEM) != cudaSuccess ||
      cudaFuncSetAttribute(k_radix_one, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)RO_SMEM) != cudaSuccess)
    return FC_ERR_CUDA;
  if (cudaMemsetAsync(ctl, 0, 64, s) != cudaSuccess) return FC_ERR_CUDA;

  // Every position by its first symbols.  The first pass reads the text itself (and checks it, before anything
  // is written to the outputs); its pairs land where the last pass ends in (key_a, d_sa).
  Sym y;
  y.bits = bits_for(vocab);
  y.count = std::min(8, 64 / y.bits);
  y.inv = (65536u + (uint32_t)y.bits - 1u) / (uint32_t)y.bits;
  const int key_bits = y.bits * y.count, np = (key_bits + 7) / 8;
  const TextKeys tx{d_tokens, y};
  k_radix_hist<true><<<(unsigned)L.nb, RS_THREADS, 0, s>>>(nullptr, tx, n, 0, hist, L.nb, vocab, ctl);
  if (!read_counts()) return FC_ERR_CUDA;
  if (hc.flag) return FC_ERR_INVALID_ARG;
  {
    uint64_t* k0 = np % 2 ? key_a : key_b;
    uint32_t* v0 = np % 2 ? d_sa : val_b;
    if (!offsets(n)) return FC_ERR_CUDA;
    if (fc_launch_dependent(k_radix_scatter<true>, dim3((unsigned)L.nb), RS_THREADS, 0, s, 0, nullptr, nullptr, tx, k0, v0, n, 0,
                            hist, L.nb) != FC_OK ||
        !passes(k0, v0, np % 2 ? key_b : key_a, np % 2 ? val_b : d_sa, n, 1, key_bits))
      return FC_ERR_CUDA;
  }
  // The sorted keys are in key_a.  key_b takes the list of small ranges (8 bytes an element, n at most), the rank
  // area the tables of longer ones; the lists alternate between key_b and key_a from then on.
  Elem* lists[2] = {reinterpret_cast<Elem*>(key_b), reinterpret_cast<Elem*>(key_a)};
  const size_t mid_cap = n / (SMALL_MAX + 1) + 1, huge_cap = n / (MID_MAX + 1) + 1;
  char* tab = reinterpret_cast<char*>(rank);
  Range* mids[2] = {reinterpret_cast<Range*>(tab), reinterpret_cast<Range*>(tab) + mid_cap};
  HugeRange* huges[2];
  huges[0] = reinterpret_cast<HugeRange*>(tab + align_up(2 * mid_cap * sizeof(Range), 16));
  huges[1] = huges[0] + huge_cap;
  // first tokens come with the keys, unless gaps of unused tokens could be long
  const bool buckets = vocab <= 65536u;
  k_split<false><<<(unsigned)cdiv(n, SPL_TILE), SPL_THREADS, 0, s>>>(key_a, d_sa, n, y, (uint32_t)y.count, nullptr, d_sa,
                                                                     d_lcp, lists[0], mids[0], huges[0], ct, 0,
                                                                     buckets ? d_bucket : nullptr, vocab);
  // Ranges of more than MID_MAX suffixes: gathered and sorted, while that makes headway.
  int hin = 0;
  uint64_t before = ~0ull;
  bool doubling = false;
  uint64_t h = (uint64_t)y.count;  // tokens that every range is known to share (some share more)
  for (;;) {
    k_huge_base<<<1, SCAN_THREADS, 0, s>>>(huges[hin], ct, hin);
    if (!read_counts()) return FC_ERR_CUDA;
    const uint32_t ng = hc.huge[hin], m = hc.total;
    if (ng == 0) break;
    Sym yh = y;
    const int obits = bits_for(ng - 1);
    yh.count = std::min(y.count, (63 - obits) / y.bits);  // the range's index lies above the symbols
    if (2ull * m > before || yh.count < 1) {
      doubling = true;
      break;
    }
    before = m;
    const int bits = yh.bits * yh.count + obits;
    uint64_t* k1 = key_b + (n - m);  // behind the list: small elements and gathered ones are n at most
    const bool odd = (bits + 7) / 8 % 2 != 0;  // the last pass ends in (key_a, val_b)
    uint64_t *kf = odd ? k1 : key_a, *kt = odd ? key_a : k1;
    uint32_t *vf = odd ? head : val_b, *vt = odd ? val_b : head;
    k_huge_gather<<<grid_for(m, 256), 256, 0, s>>>(d_tokens, n, yh, d_sa, huges[hin], ng, m, kf, vf);
    if (!passes(kf, vf, kt, vt, m, 0, bits)) return FC_ERR_CUDA;
    k_split<true><<<(unsigned)cdiv(m, SPL_TILE), SPL_THREADS, 0, s>>>(key_a, val_b, m, yh, (uint32_t)yh.count, huges[hin],
                                                                      d_sa, d_lcp, lists[0], mids[0], huges[hin ^ 1], ct,
                                                                      hin ^ 1, nullptr, 0u);
    hin ^= 1;
  }
  // Rounds of y.count more tokens over the rest.
  const int sms = std::max(1, sm_count());
  int round = 0, check = 0;
  unsigned long long mid_before = 0;  // mid_work after the first two rounds
  while (!doubling) {
    const int in = round % 3;
    if (round == check) {
      if (round && !read_counts()) return FC_ERR_CUDA;
      if (hc.small[in] == 0 && hc.mid[in] == 0) break;
      if (round == 2) mid_before = hc.mid_work;
      // Most suffixes still together after six rounds, or 34 rounds; or mid ranges that stay (a text of hundreds of
      // tokens in many copies): sorting n / 2 suffixes of theirs takes as long as a round of doubling.  5M tokens, ms,
      // doubling from the start / without this line / n suffixes / n / 2 / n / 4: 3000 copies of 200 tokens 5.2 / 5.7 /
      // 4.3 / 4.3 / 3.8, of 100 4.6 / 3.2 / 3.2 / 3.3 / 3.1, 100 of 3000 8.0 / 8.6 / 8.4 / 6.9 / 6.6; 50M tokens, 3000
      // of 400 73 / 32 / 32 / 31 / 35.
      if (round >= 32 || (round >= 6 && (hc.small[in] > n / 4 || (hc.mid[in] && hc.mid_work - mid_before > n / 2)))) {
        doubling = true;
        break;
      }
      check = round ? round + 4 : 2;
    }
    const int o = (round + 1) % 3, li = round & 1;
    const int many = round == 0 ? 1 : 8;
    const unsigned gs = (unsigned)std::min<uint64_t>(cdiv(n, RFS_HEADS), 8ull * sms), gm = 4u * sms;
    if (fc_launch_dependent(k_refine_small, dim3(gs), RFS_THREADS, 0, s, 0, d_tokens, n, y, d_sa, d_lcp, lists[li],
                            lists[li ^ 1], ct, in, o, many) != FC_OK ||
        fc_launch_dependent(k_refine_mid, dim3(gm), RFM_THREADS, RFM_SMEM, s, 0, d_tokens, n, y, d_sa, d_lcp, mids[li],
                            mids[li ^ 1], lists[li ^ 1], ct, in, o) != FC_OK)
      return FC_ERR_CUDA;
    ++round;
    h += (uint64_t)y.count;
  }
  if (doubling) {
    // The ranks go where the tables are not; from then on the two areas have changed places.
    k_rank_slots<<<g, 256, 0, s>>>(d_sa, n, head);
    k_rank_ranges<<<grid_for(n, 256), 256, 0, s>>>(d_sa, lists[round & 1], mids[round & 1], huges[hin], ct, round % 3, hin,
                                                   head);
    std::swap(rank, head);
    for (int r = 0;; ++r) {
      if (r > 40 || h >= 4 * n + 64) return FC_ERR_INTERNAL;
      k_keys_round<<<g, 256, 0, s>>>(d_sa, rank, n, h, key_a, d_sa);
      // LSD passes over the populated bits of the low then the high word
      uint64_t* kin = key_a;
      uint32_t* vin = d_sa;
      uint64_t* kout = key_b;
      uint32_t* vout = val_b;
      int shifts[16];
      int np = 0;
      for (int b = 0; b < bits_for(n); b += 8) shifts[np++] = b;
      for (int b = 0; b < bits_for(n - 1); b += 8) shifts[np++] = 32 + b;
      for (int p = 0; p < np; ++p) {
        if (!pass(kin, vin, kout, vout, n, shifts[p])) return FC_ERR_CUDA;
        std::swap(kin, kout);
        std::swap(vin, vout);
      }
      // kin/vin now hold the sorted keys and positions.
      k_heads<<<g, 256, 0, s>>>(kin, n, head);
      if (exclusive_scan(head, n, stmp, s) != cudaSuccess) return FC_ERR_CUDA;
      k_ranks<<<g, 256, 0, s>>>(kin, vin, head, n, rank, d_sa, ctl);
      if (!read_counts()) return FC_ERR_CUDA;
      if (hc.groups == n) break;
      if (hc.groups == 0 || hc.groups > n) return FC_ERR_INTERNAL;
      h *= 2;
    }
    // every group is a single suffix now, so rank is the inverse suffix array
    k_lcp<<<g, 256, 0, s>>>(d_tokens, d_sa, rank, n, d_lcp);
  }
  if (!buckets) k_bucket<<<grid_for((uint64_t)vocab + 1, 256), 256, 0, s>>>(d_tokens, d_sa, n, vocab, d_bucket);
  if (cudaGetLastError() != cudaSuccess) return FC_ERR_CUDA;
  if (cudaStreamSynchronize(s) != cudaSuccess) return FC_ERR_CUDA;
  if (out) {
    out->tokens = d_tokens;
    out->sa = d_sa;
    out->bucket = d_bucket;
    out->lcp = d_lcp;
    out->n_tokens = n;
    out->vocab = vocab;
    out->keys = nullptr;
  }
  return FC_OK;
}

// ---------------------------------------------------------------------------
// Datastore build without any allocation: the scratch space lives in a
// fixed array compiled into this library instead of caller memory.
//
// Some callers cannot call cudaMalloc: a serving process whose memory manager
// reserves all free device memory for its KV cache up front (a later
// cudaMalloc fails, or fragments that reservation), or a plugin inside a host
// application that owns every device allocation.  They can still build a
// small datastore (a repository's own project store) here.
//
// The array is a file-scope __device__ variable.  A GPU holds it from the
// moment this file's device code is loaded there until the process exits.
// Under CUDA's default lazy module loading that moment is the first datastore
// build (this entry point or fc_datastore_build) made on the device, not the
// library's load: the first call itself places the 30 MiB.  A caller that
// reserves all free device memory must therefore make one call (a small
// corpus is enough) before reserving it.
//
// Host code cannot pass the variable's name to a kernel (on the host it is
// only a stand-in, not a device address): every call looks up the device
// address on the current device with cudaGetSymbolAddress.  The lookup is
// not cached, so the address stays right after a device reset reloads the
// module elsewhere.  The first call on a device loads the module, so it
// should come before any stream capture.  Every call shares the one array
// and leaves its contents behind; the build clears what must start at zero
// itself.  Calls whose work overlaps on the GPU (two streams, two host
// threads) race on the array and must not be made.
// ---------------------------------------------------------------------------
namespace {
constexpr size_t kNoAllocScratchBytes = (size_t)30 << 20;  // 30 MiB
static __device__ __align__(256) unsigned char g_sa_scratch[kNoAllocScratchBytes];

fc_status scratch_for_current_device(void** out) {
  void* p = nullptr;
  if (cudaGetSymbolAddress(&p, g_sa_scratch) != cudaSuccess || !p) return FC_ERR_CUDA;
  *out = p;
  return FC_OK;
}
}  // namespace

extern "C" fc_status fc_datastore_build_noalloc(const uint32_t* d_tokens, uint64_t n_tokens, uint32_t vocab,
                                                uint32_t* d_sa, uint32_t* d_bucket, uint8_t* d_lcp,
                                                fc_stream stream, fc_datastore* out) {
  FC_NVTX_RANGE();
  if (n_tokens > FC_NOALLOC_MAX_TOKENS) return FC_ERR_CAPACITY;
  if (n_tokens > 0 && fc_datastore_build_workspace(n_tokens, vocab) > kNoAllocScratchBytes) return FC_ERR_CAPACITY;
  void* ws = nullptr;
  fc_status st = scratch_for_current_device(&ws);
  if (st != FC_OK) return st;
  return fc_datastore_build(d_tokens, n_tokens, vocab, d_sa, d_bucket, d_lcp, ws, kNoAllocScratchBytes, stream, out);
}

// ---------------------------------------------------------------------------
// Suffix keys: entry j = (sa[j], T[sa[j] + 1 .. sa[j] + 7]), FC_PAD_TOKEN past
// the corpus end; 32 bytes, written as two 16-byte stores.
// ---------------------------------------------------------------------------
namespace {
// VEC: the corpus is 16-byte aligned, and a suffix's tokens 1..7 come from the
// aligned 16-byte groups they lie in (all inside the corpus) instead of seven
// 4-byte loads.  Bound by the random reads: 20M tokens 352 us with 4-byte loads
// alone, 283 us now.
template <bool VEC>
__global__ void k_suffix_keys(const uint32_t* __restrict__ T, const uint32_t* __restrict__ sa, uint64_t n,
                              uint4* __restrict__ keys) {
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t j = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; j < n; j += stride) {
    const uint64_t i = __ldg(sa + j);
    uint32_t t[8];
    t[0] = (uint32_t)i;
    const uint64_t g = (i + 1) >> 2;  // the group of token i + 1
    if (VEC && 4 * (g + 3) <= n) {
      const uint4* Tv = reinterpret_cast<const uint4*>(T) + g;
      const int o = (int)(i + 1) & 3;
      const uint4 a = __ldg(Tv), b = __ldg(Tv + 1), c = o > 1 ? __ldg(Tv + 2) : make_uint4(0, 0, 0, 0);
      const uint32_t w[10] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w, c.x, c.y};
#pragma unroll
      for (int k = 0; k < 7; ++k) t[k + 1] = o == 0 ? w[k] : o == 1 ? w[k + 1] : o == 2 ? w[k + 2] : w[k + 3];
    } else {
#pragma unroll
      for (int k = 1; k < 8; ++k) t[k] = (i + k < n) ? __ldg(T + i + k) : FC_PAD_TOKEN;
    }
    keys[2 * j] = make_uint4(t[0], t[1], t[2], t[3]);
    keys[2 * j + 1] = make_uint4(t[4], t[5], t[6], t[7]);
  }
}
}  // namespace

extern "C" fc_status fc_datastore_keys(const fc_datastore* ds, uint32_t* d_keys, fc_stream stream) {
  FC_NVTX_RANGE();
  if (!ds || !ds->tokens || !ds->sa || !d_keys || ds->n_tokens == 0 || ds->n_tokens >= 0xFFFFFFFFull)
    return FC_ERR_INVALID_ARG;
  if (reinterpret_cast<uintptr_t>(d_keys) % 32) return FC_ERR_INVALID_ARG;
  const uint64_t n = ds->n_tokens;
  const auto kern = reinterpret_cast<uintptr_t>(ds->tokens) % 16 == 0 ? k_suffix_keys<true> : k_suffix_keys<false>;
  kern<<<grid_for(n, 256), 256, 0, static_cast<cudaStream_t>(stream)>>>(ds->tokens, ds->sa, n,
                                                                        reinterpret_cast<uint4*>(d_keys));
  return FC_CHECK_LAUNCH();
}

// ---------------------------------------------------------------------------
// The reversed corpus R[i] = T[n-1-i], whose suffix array serves
// fc_retrieve_rev.  Aligned 16-byte groups where both sides allow it: output
// group q (tokens 4q .. 4q+3) reads input tokens n-4-4q .. n-1-4q, which are
// 16-byte aligned exactly when n is a multiple of 4.
// ---------------------------------------------------------------------------
namespace {
__global__ void k_reverse(const uint32_t* __restrict__ in, uint64_t n, uint32_t* __restrict__ out) {
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  const uint64_t t0 = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
  const bool vec = (n % 4 == 0) && (reinterpret_cast<uintptr_t>(in) % 16 == 0) &&
                   (reinterpret_cast<uintptr_t>(out) % 16 == 0);
  if (vec) {
    const uint64_t groups = n / 4;
    for (uint64_t q = t0; q < groups; q += stride) {
      const uint4 v = __ldg(reinterpret_cast<const uint4*>(in) + (groups - 1 - q));
      reinterpret_cast<uint4*>(out)[q] = make_uint4(v.w, v.z, v.y, v.x);
    }
  } else {
    for (uint64_t i = t0; i < n; i += stride) out[i] = __ldg(in + (n - 1 - i));
  }
}
}  // namespace

extern "C" fc_status fc_reverse_tokens(const uint32_t* d_tokens, uint64_t n_tokens, uint32_t* d_out,
                                       fc_stream stream) {
  FC_NVTX_RANGE();
  if (n_tokens == 0) return FC_OK;
  if (!d_tokens || !d_out || d_tokens == d_out || n_tokens >= 0xFFFFFFFFull) return FC_ERR_INVALID_ARG;
  const uint64_t a = reinterpret_cast<uintptr_t>(d_tokens), b = reinterpret_cast<uintptr_t>(d_out);
  if (a < b + 4 * n_tokens && b < a + 4 * n_tokens) return FC_ERR_INVALID_ARG;  // overlapping buffers
  k_reverse<<<grid_for(cdiv(n_tokens, 4), 256), 256, 0, static_cast<cudaStream_t>(stream)>>>(d_tokens, n_tokens,
                                                                                            d_out);
  return FC_CHECK_LAUNCH();
}
