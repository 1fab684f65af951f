// Hilbert sort: stable LSD radix sort of the K-word key prefixes, then the
// fix-up that orders runs of equal prefixes by full key.
//
// Paper, Section 2: the Hilbert order is a total order over the points; the
// paper sorts with a key-free CPU algorithm whose details it does not give.
// Here the order is "ascending (full key, point index)": the prefix words are
// sorted with 8-bit digits, least significant first; each pass is one
// single-pass binning kernel with decoupled look-back (Merrill & Garland 2016;
// Adinets & Merrill 2022, "Onesweep"). The input starts in point order, so
// equal prefixes stay in index order; the fix-up then reorders each run of
// equal prefixes by its full keys.
//
// The trees of a batch are sorted together: one launch per pass covers every
// tree, and tile tickets interleave the trees (ticket g is tile g / TB of tree
// g % TB), so the tiles in flight at any time are spread over all trees and
// each tree's look-back chain stays short.
//
// The look-back is the only wait between blocks. Tiles take tickets from an
// atomic counter, so a tile only ever waits for tiles that started before it;
// each wait is bounded by a %globaltimer deadline, after which the tile sets
// the error word (HF_ETIMEOUT), publishes a value and finishes.
#include <cuda_runtime.h>

#include <algorithm>
#include <vector>

#include "hf_internal.cuh"
#include "hilbert_device.cuh"

namespace {

constexpr int NT = 256;
constexpr int IPT = 8;
constexpr int TILE = NT * IPT;  // 2048 keys per tile
constexpr int WARPS = NT / 32;
constexpr uint32_t FLAG_AGG = 1u << 30;
constexpr uint32_t FLAG_PRE = 2u << 30;
constexpr uint32_t VAL_MASK = (1u << 30) - 1u;
constexpr int LB = 16;  // predecessor status words read per look-back round

__device__ __forceinline__ uint32_t ld_relaxed(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_relaxed(uint32_t* p, uint32_t v) {
  asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ uint64_t globaltimer() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ uint32_t lanemask_lt() {
  uint32_t m;
  asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
  return m;
}

// Digit histograms of all 8 bytes of all K prefix words (order-independent).
// Tree blockIdx.y: keys at pk + y * pk_ts, histograms at hist + y * K * 8 * 256.
__global__ void digit_hist_kernel(const uint64_t* __restrict__ pk, int64_t pk_ts, int64_t n, int K,
                                  uint32_t* __restrict__ hist) {
  extern __shared__ uint32_t sh[];  // [K*8][256]
  pk += blockIdx.y * pk_ts;
  hist += (size_t)blockIdx.y * K * 8 * 256;
  const int nh = K * 8 * 256;
  for (int i = threadIdx.x; i < nh; i += blockDim.x) sh[i] = 0;
  __syncthreads();
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n;
       e += (int64_t)gridDim.x * blockDim.x) {
    for (int w = 0; w < K; ++w) {
      const uint64_t key = __ldg(pk + (size_t)w * n + e);
#pragma unroll
      for (int b = 0; b < 8; ++b) atomicAdd(&sh[(w * 8 + b) * 256 + ((key >> (8 * b)) & 255)], 1u);
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < nh; i += blockDim.x)
    if (sh[i]) atomicAdd(&hist[i], sh[i]);
}

// Exclusive scan of each 256-bin histogram (one block per histogram).
__global__ void hist_scan_kernel(uint32_t* __restrict__ hist) {
  __shared__ uint32_t s[256];
  uint32_t* h = hist + blockIdx.x * 256;
  s[threadIdx.x] = h[threadIdx.x];
  __syncthreads();
  if (threadIdx.x == 0) {
    uint32_t run = 0;
    for (int i = 0; i < 256; ++i) {
      const uint32_t c = s[i];
      s[i] = run;
      run += c;
    }
  }
  __syncthreads();
  h[threadIdx.x] = s[threadIdx.x];
}

// ---------------------------------------------------------------------------
// How many of the low digits a tree's sort can leave out. On most data a
// prefix of 32 to 64 bits already tells nearly all points apart, and the few
// runs that share it are cheaper to order by counting (refine_warp_kernel)
// than by the passes over every point that the remaining digits cost. The
// runs' sizes are estimated from a sample: C pairs of equal top bits among S
// points mean about n + 2 C (n / S)^2 word compares in the ranking. One block
// per tree sorts S evenly spread, jittered points' first words and prices the
// choices: start at pass 0 (every digit of the K <= 2 words), or order by the
// first word's top 64, 56, 48, 40 or 32 bits.
// Prices in picoseconds (3M x 384, 4M x 64, 1.2M x 128): a pass 11 per point
// (or its launch's latency, on small inputs), refining 24 per point and 60 per
// point of a run that reaches past a warp's 32 positions, a compare 0.5,
// fetching the first word again in the final order 9. The members of the longest
// run wait for a chain of as many compares, 120 ns each (40 where the first
// words are equal and only the second ones are read), once for all trees of the
// batch, which is the refining's time where it is above the rest (50,000 x 384
// mixture data, T = 1, without this price: runs of up to 1,731, 207 us of
// refining to save 104 us of passes). A run that the sample misses costs time,
// not order. Per sort: 3M x 384, T = 64: 33.2 -> 25.9 ms of
// kernels; 4M x 64, T = 16, where half of the points tie at 128 bits, keeps
// every pass; 200,001 x 384, T = 16: 3.88 -> 3.74 ms, build and narrow graph.
// A sample of 4096 takes 70 us, one block's sort, and one of 1024 24 us, which
// misjudges the runs of large inputs (3M x 384: 6.7 ms lost, 4M x 64: 2.5).
// ---------------------------------------------------------------------------
constexpr int64_t PLAN_LARGE = (int64_t)1 << 18;  // points from which the sample is 4096
constexpr int PLAN_LEVELS = 5;

template <int PLAN_S>
__global__ void __launch_bounds__(1024) sort_plan_kernel(const uint64_t* __restrict__ pk, int64_t pk_ts, int64_t n,
                                                         int K, int TB, uint32_t* __restrict__ skip,
                                                         uint32_t* __restrict__ first) {
  constexpr int E = PLAN_S / 1024;
  __shared__ uint64_t s[PLAN_S];
  __shared__ unsigned long long pairs[PLAN_LEVELS];
  __shared__ uint32_t longest[PLAN_LEVELS];
  const uint64_t* word = pk + blockIdx.x * pk_ts;
  const int tid = threadIdx.x;
  const int S = n < PLAN_S ? (int)n : PLAN_S;
  // bitonic sort of element e * 1024 + tid in register e, padded with the
  // largest word: partners less than 32 apart by shuffles
  uint64_t v[E];
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const int j = e * 1024 + tid;
    const uint32_t h = (uint32_t)j * 0x9E3779B1u;
    const int64_t a = n * j / S, b = n * (j + 1) / S;  // this sample's share of the points
    v[e] = j < S ? __ldg(word + a + (int64_t)((h >> 8) % (uint64_t)(b - a))) : ~0ull;
  }
  if (tid < PLAN_LEVELS) pairs[tid] = longest[tid] = 0;
#pragma unroll 1
  for (int kk = 2; kk <= PLAN_S; kk <<= 1)
#pragma unroll 1
    for (int j = kk >> 1; j > 0; j >>= 1) {
      if (j >= 32) {
        __syncthreads();
#pragma unroll
        for (int e = 0; e < E; ++e) s[e * 1024 + tid] = v[e];
        __syncthreads();
      }
#pragma unroll
      for (int e = 0; e < E; ++e) {
        const int i = e * 1024 + tid;
        const uint64_t o = j >= 32 ? s[i ^ j] : __shfl_xor_sync(0xffffffffu, v[e], j);
        const bool small = ((i & kk) == 0) == ((i & j) == 0);  // this place keeps the smaller
        if (small ? o < v[e] : o > v[e]) v[e] = o;
      }
    }
  __syncthreads();
#pragma unroll
  for (int e = 0; e < E; ++e) s[e * 1024 + tid] = v[e];
  __syncthreads();
  for (int l = 0; l < PLAN_LEVELS; ++l) {
    unsigned long long mine = 0;
    uint32_t most = 0;  // points before one that share its top bits
    for (int i = tid; i < S; i += 1024) {  // (padding sorts last)
      const uint64_t v = s[i] >> (8 * l);
      int lo = 0, hi = i;  // first point with these top bits
      while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if ((s[mid] >> (8 * l)) < v) lo = mid + 1;
        else hi = mid;
      }
      mine += (unsigned long long)(i - lo);
      most = max(most, (uint32_t)(i - lo));
    }
    most = __reduce_max_sync(0xffffffffu, most);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mine += __shfl_down_sync(0xffffffffu, mine, o);
    if ((tid & 31) == 0 && mine) {
      atomicAdd(&pairs[l], mine);
      atomicMax(&longest[l], most);
    }
  }
  __syncthreads();
  if (tid == 0) {
    const double dn = (double)n, grow = (dn / S) * (dn / S);
    const double pass = fmax(11.0 * dn, 8e6 / TB);  // a launch takes 8 us at least, shared by the trees
    double best = pass * 8 * K;
    uint32_t s0 = 0;
    for (int l = 0; l < PLAN_LEVELS; ++l) {
      const double compares = 2.0 * (double)pairs[l] * grow;
      // mates per point; a run of m crosses a 32-position boundary with
      // probability about m / 32
      const double mates = compares / dn, cross = mates / (mates + 32.0);
      // (two samples of one run may be all of it)
      const double chain = longest[l] > 1 ? (l ? 120e3 : 40e3) * (longest[l] - 1) * (dn / S) / TB : 0.0;
      const double cost =
          pass * (8 - l) + 24.0 * dn + fmax(cross * (60.0 * dn + 0.5 * compares), chain) + (l ? 9.0 * dn : 0.0);
      const uint32_t st = (uint32_t)(8 * (K - 1) + l);
      if (st && cost < best) {
        best = cost;
        s0 = st;
      }
    }
    skip[blockIdx.x] = first[blockIdx.x] = s0;
    atomicMax(&skip[TB], 255u - s0);
  }
}

struct PassSmem {
  uint64_t keys[TILE];
  uint32_t vals[TILE];
  uint32_t whist[WARPS][256];
  uint32_t tile_start[256];
  uint32_t gbase[256];
  uint32_t scan[WARPS];
  uint32_t tile;
};

// One pass over the trees of a batch. Each array is given as the first
// tree's pointer plus the element stride between trees.
struct PassArgs {
  const uint64_t* keys_in;
  int64_t keys_in_ts;
  const uint32_t* vals_in;
  int64_t vals_in_ts;
  const uint64_t* gather_src;
  int64_t gather_src_ts;
  uint64_t* keys_out;
  int64_t keys_out_ts;
  uint32_t* vals_out;
  int64_t vals_out_ts;
  const uint32_t* goff;  // exclusive digit offsets of this pass
  int64_t goff_ts;
  uint32_t* status;      // [TB][ntiles + 1][256]
  uint32_t* ticket;
  int* err;
  int64_t n, ntiles;
  uint64_t spin_ns;
  int shift, TB, stall;
  // first pass of each tree, then 255 less the least of them (0: every pass
  // runs, as without the array);
  // a tree's first pass reads the digit's word in point order
  const uint32_t* skip;
  const uint64_t* first_src;
  int64_t first_src_ts;
  uint32_t pass;
};

// One LSD pass: bins the keys of one tile by `digit = key >> shift & 255`.
// GATHER: the key of the element at position e is gather_src[vals_in[e]]
// (the next prefix word, fetched in the current order).
template <bool GATHER>
__global__ void __launch_bounds__(NT, 5) onesweep_kernel(const PassArgs a) {
  extern __shared__ __align__(16) unsigned char smraw[];
  PassSmem& S = *reinterpret_cast<PassSmem*>(smraw);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (a.skip) {
    const uint32_t least = __ldg(a.skip + a.TB);
    if (least && a.pass < 255u - least) return;  // no tree needs this digit
  }

  if (tid == 0) S.tile = atomicAdd(a.ticket, 1u);
  for (int i = tid; i < WARPS * 256; i += NT) (&S.whist[0][0])[i] = 0;
  __syncthreads();
  const int64_t tr = S.tile % (uint32_t)a.TB;
  const int64_t tile = S.tile / (uint32_t)a.TB;
  const int64_t n = a.n, ntiles = a.ntiles;
  const int shift = a.shift;
  const uint32_t s0 = a.skip ? __ldg(a.skip + tr) : 0u;
  if (a.pass < s0) return;
  // a tree's first pass reads the word in point order (vals_in null: identity)
  const bool first = a.skip && a.pass == s0;
  const uint32_t* __restrict__ vals_in = first ? nullptr : a.vals_in + tr * a.vals_in_ts;
  const uint64_t* __restrict__ src = first    ? a.first_src + tr * a.first_src_ts
                                     : GATHER ? a.gather_src + tr * a.gather_src_ts
                                              : a.keys_in + tr * a.keys_in_ts;
  uint64_t* __restrict__ keys_out = a.keys_out + tr * a.keys_out_ts;
  uint32_t* __restrict__ vals_out = a.vals_out + tr * a.vals_out_ts;
  const uint32_t* __restrict__ goff = a.goff + tr * a.goff_ts;
  uint32_t* __restrict__ status = a.status + (size_t)tr * (ntiles + 1) * 256;
  int* err = a.err;
  const int64_t base = tile * TILE;

  uint64_t k[IPT];
  uint32_t v[IPT];
  uint32_t rk[IPT];
  uint32_t dg[IPT];
#pragma unroll
  for (int j = 0; j < IPT; ++j) {
    const int64_t e = base + warp * 32 * IPT + j * 32 + lane;
    if (e < n) {
      // read once per pass: streaming loads leave L2 to the pass's output
      v[j] = vals_in ? __ldcs(vals_in + e) : (uint32_t)e;
      if (GATHER && vals_in) {
        // values are point indices < n unless an earlier pass gave up its
        // look-back (error word set); never read outside the source then
        if (v[j] >= (uint64_t)n) {
          hf_raise(err, HF_ERRBIT_TIMEOUT);
          v[j] = 0;
        }
        k[j] = __ldg(src + v[j]);
      } else {
        k[j] = __ldcs(reinterpret_cast<const unsigned long long*>(src) + e);
      }
      dg[j] = (uint32_t)(k[j] >> shift) & 255u;
    } else {
      v[j] = 0;
      k[j] = 0;
      dg[j] = 256u;  // sentinel: no element
    }
  }
  // Stable ranking within the warp: items are ordered by (j, lane).
  const uint32_t lt = lanemask_lt();
#pragma unroll
  for (int j = 0; j < IPT; ++j) {
    const uint32_t peers = __match_any_sync(0xffffffffu, dg[j]);
    const uint32_t before = __popc(peers & lt);
    uint32_t basec = 0;
    if (dg[j] < 256u) basec = S.whist[warp][dg[j]];
    __syncwarp();
    if (dg[j] < 256u && before == 0) S.whist[warp][dg[j]] = basec + __popc(peers);
    __syncwarp();
    rk[j] = basec + before;
  }
  __syncthreads();

  // Per digit: exclusive offsets across warps and the tile's count.
  const int dgt = tid;  // NT == 256 == radix
  uint32_t cnt = 0;
#pragma unroll
  for (int w = 0; w < WARPS; ++w) {
    const uint32_t c = S.whist[w][dgt];
    S.whist[w][dgt] = cnt;
    cnt += c;
  }

  // The tile's counts are published first (its successors can use them at
  // once); the tile-local offsets and the scatter into shared memory run
  // before this tile waits for its own predecessors.
  uint32_t* st = status + tile * 256 + dgt;
  st_relaxed(st, (tile == 0 ? FLAG_PRE : FLAG_AGG) | cnt);

  // Tile-local exclusive scan of the digit counts (warp scans + warp totals),
  // folded into the per-warp offsets.
  uint32_t incl = cnt;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  if (lane == 31) S.scan[warp] = incl;
  __syncthreads();
  uint32_t woff = 0;
#pragma unroll
  for (int w = 0; w < WARPS; ++w)
    if (w < warp) woff += S.scan[w];
  const uint32_t tstart = woff + incl - cnt;
  S.tile_start[dgt] = tstart;
#pragma unroll
  for (int w = 0; w < WARPS; ++w) S.whist[w][dgt] += tstart;
  __syncthreads();

  // Scatter into shared memory in digit order.
#pragma unroll
  for (int j = 0; j < IPT; ++j) {
    if (dg[j] < 256u) {
      const uint32_t lp = S.whist[warp][dg[j]] + rk[j];
      S.keys[lp] = k[j];
      S.vals[lp] = v[j];
    }
  }

  // Decoupled look-back for this digit. LB predecessor status words are read
  // at once (independent loads, one round trip), then consumed in order:
  // aggregates are added until an inclusive prefix ends the walk; a word that
  // is not ready yet is re-read from there on the next round.
  uint32_t excl = 0;
  if (tile > 0) {
    int64_t pred = tile - 1;
    const uint64_t t0 = globaltimer();
    uint32_t spins = 0;
    for (;;) {
      uint32_t sv[LB];
#pragma unroll
      for (int i = 0; i < LB; ++i) {
        // test hook: tile 1 watches the spare status row that nothing writes
        const int64_t pt = pred - i;
        const uint32_t* ps = (a.stall && tr == 0 && tile == 1) ? status + ntiles * 256 + dgt : status + pt * 256 + dgt;
        sv[i] = pt >= 0 ? ld_relaxed(ps) : FLAG_PRE;  // before tile 0: prefix 0
      }
      int used = 0;
      bool done = false;
#pragma unroll
      for (int i = 0; i < LB; ++i) {
        if (used != i) break;  // stopped at an earlier word
        const uint32_t flag = sv[i] & ~VAL_MASK;
        if (flag == 0) break;
        excl += sv[i] & VAL_MASK;
        ++used;
        if (flag == FLAG_PRE) {
          done = true;
          break;
        }
      }
      if (done) break;
      pred -= used;
      if (used == 0 && (++spins & 15u) == 0 && (globaltimer() - t0 > a.spin_ns || spins > (1u << 28))) {
        hf_raise(err, HF_ERRBIT_TIMEOUT);
        break;
      }
    }
    st_relaxed(st, FLAG_PRE | ((excl + cnt) & VAL_MASK));
  }
  S.gbase[dgt] = goff[dgt] + excl;
  __syncthreads();

  // Write out coalesced (runs of equal digits go to consecutive positions).
  const int valid = (int)(n - base < TILE ? n - base : TILE);
  for (int e = tid; e < valid; e += NT) {
    const uint64_t key = S.keys[e];
    const uint32_t dgi = (uint32_t)(key >> shift) & 255u;
    const uint32_t pos = S.gbase[dgi] + (uint32_t)e - S.tile_start[dgi];
    keys_out[pos] = key;
    vals_out[pos] = S.vals[e];
  }
}

// Sorted prefix words: out[w][p] = pk[w][sigma[p]], w = 1 .. K-1, and word 0
// of the trees that were not sorted by all of it. Tree blockIdx.y of the batch
// (one launch for all of them).
__global__ void gather_prefix_kernel(const uint64_t* __restrict__ pk0, int64_t pk_ts,
                                     const uint32_t* __restrict__ sigma0, int64_t n, int K,
                                     const uint32_t* __restrict__ skip, uint64_t* __restrict__ out0,
                                     const int* __restrict__ err) {
  if (*(volatile const int*)err) return;  // the order is not valid: skip
  const int w0 = __ldg(skip + blockIdx.y) > 8u * (K - 1) ? 0 : 1;
  if (w0 >= K) return;
  const uint64_t* pk = pk0 + blockIdx.y * pk_ts;
  const uint32_t* sigma = sigma0 + blockIdx.y * n;
  uint64_t* out = out0 + (size_t)blockIdx.y * K * n;
  for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < n;
       p += (int64_t)gridDim.x * blockDim.x) {
    const uint32_t i = sigma[p];
    if (i >= (uint64_t)n) continue;
    for (int w = w0; w < K; ++w) out[(size_t)w * n + p] = __ldg(pk + (size_t)w * n + i);
  }
}

__device__ __forceinline__ bool prefix_eq(const uint64_t* __restrict__ pre, int64_t n, int K,
                                          int64_t a, int64_t b) {
  for (int w = 0; w < K; ++w)
    if (__ldg(pre + (size_t)w * n + a) != __ldg(pre + (size_t)w * n + b)) return false;
  return true;
}

__device__ __forceinline__ bool full_less(const uint64_t* a, uint32_t ia, const uint64_t* b,
                                          uint32_t ib, int W) {
  for (int w = 0; w < W; ++w)
    if (a[w] != b[w]) return a[w] < b[w];
  return ia < ib;
}

// Running XOR from the most significant bit down: bit j of the result is the
// XOR of bits 31..j of v.
__device__ __forceinline__ uint32_t xor_scan_msb(uint32_t v) {
  v ^= v >> 1;
  v ^= v >> 2;
  v ^= v >> 4;
  v ^= v >> 8;
  v ^= v >> 16;
  return v;
}

// ---------------------------------------------------------------------------
// Runs of equal prefixes (the LSD passes left each run in index order). Three
// launches cover every tree of the batch (tree blockIdx.y), with one thread
// per tied position rather than one block per run: a run has about ten members
// on clustered data, and a block that holds one run at a time keeps a handful
// of its lanes busy (4M x 64, T = 16, mixture data with about half of the
// points tied at 128 bits: 393 ms of kernels in that form; the whole build went
// from 337 to 20.4 ms, and one of 1.2M x 128 rows with few ties lost 0.8 ms of
// its 32 small launches).
//   tie_mark   finds the tied positions, lists them, keeps their points and
//              the first key word past the prefix (word K) where that is cheap;
//   tie_words  word K by the transform of the top Lf levels, for the rest;
//   tie_rank   each member counts the members of its run that precede it.
// Members that also tie on every word at hand form sub-runs of the ranked
// order; tie_hard orders those by the next words of the top bit level, where the
// key has any, and then by the full key. Runs longer than TIE_RUN_CAP and
// sub-runs longer than tie_hard_cap go to the list of big runs, which the host
// settles after the build's sync.
// The scratch is the sort's own, free after the last pass: words in keys_a,
// sub-runs in keys_b, points in vals_a, listed positions in vals_b.
// ---------------------------------------------------------------------------
// A member's rank costs one pass over its run: 2^26 word compares for a run at
// the cap, about 20 us of the whole chip.
constexpr int TIE_RUN_CAP = 8192;
// Sub-run members whose full keys fit a block's scratch slice: 304 slices of
// 256 x 48 words at d = 384 are 30 MB, of 256 x 128 words at d = 1024 80 MB;
// longer keys keep 64.
__host__ __device__ constexpr int tie_hard_cap(int W) { return W <= 128 ? 256 : 64; }
constexpr int TIE_HARD_WARPS = 8;
constexpr int TIE_TOP_WORDS = 3;  // words past word K that tie_hard takes from the top bit level

struct TieArgs {  // the first tree of the batch; strides below
  const uint64_t* prefix;  // [tb][K][n] sorted
  const uint64_t* pk;      // [tb][K2][n] key words, point order
  uint32_t* sigma;         // [tb][n]
  uint64_t* word;          // [tb][n] word K by position
  uint2* hard;             // [tb][n] sub-runs (start, len)
  uint32_t* pt;            // [tb][n] points by position (the order before the fix-up)
  uint32_t* list;          // [tb][n] tied positions
  uint2* big;              // [tb][big_cap]
  uint32_t* counters;      // [tb][4]: listed positions, big runs, sub-runs
  const uint32_t* skip;    // [tb] first pass of each tree's sort
  const uint32_t* planes;
  const int32_t* pi;       // [tb][d]
  const uint32_t* rbits;   // [tb][W32]
  const int* err;
  int64_t n, big_cap;
  int d, W32, bits, W, K, K2, Lf, tb, stride;
  int top;   // words K + 1 .. K + top lie in the top bit level and tie_hard tries them first
  int rows;  // coordinate rows of a tie_hard block's shared memory
};

// Key words w0 .. w0 + nw - 1 (nw <= N) of the point whose plane-0 row is `row`,
// all in the top bit level (d >= 64 (w0 + nw)): the whole warp forms them with
// ballots over the permuted, reflected top bits, carrying the parity of the
// first 64 w0. Every lane gets them.
template <int N>
__device__ __forceinline__ void tie_top_words(const uint32_t* __restrict__ row, const int32_t* __restrict__ pi,
                                              const uint32_t* __restrict__ rb, int w0, int nw, int lane,
                                              uint64_t* out) {
  auto ballot = [&](int h) {
    const int c = __ldg(pi + 32 * h + lane);
    const uint32_t bit = ((__ldg(row + (c >> 5)) >> (c & 31)) ^ (__ldg(rb + h) >> lane)) & 1u;
    return __ballot_sync(0xffffffffu, bit);
  };
  uint32_t carry = 0;
  for (int h = 0; h < 2 * w0; ++h) carry ^= __popc(ballot(h)) & 1u;
#pragma unroll
  for (int i = 0; i < N; ++i) {
    out[i] = 0;
    if (i < nw) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        uint32_t v = xor_scan_msb(__brev(ballot(2 * (w0 + i) + h)));
        if (carry) v = ~v;
        carry = v & 1u;
        out[i] = (out[i] << 32) | v;
      }
    }
  }
}

// WORDS: where word K comes from. 0: the key kernel computed it (K2 > K); 1:
// it lies in the top bit level (d >= 64 (K + 1)), a warp forms it per tied
// point with ballots over the permuted, reflected top bits, carrying the
// parity of the first 64 K; 2: tie_words.
template <int WORDS>
__global__ void __launch_bounds__(256) tie_mark_kernel(const TieArgs a) {
  if (*(volatile const int*)a.err) return;  // the order is not valid: skip
  const int64_t n = a.n;
  const int K = a.K, lane = threadIdx.x & 31;
  const size_t tr = blockIdx.y;
  const uint64_t* __restrict__ pre = a.prefix + tr * K * n;
  const uint64_t* __restrict__ pkw = a.pk + tr * a.K2 * n + (size_t)K * n;
  const uint32_t* __restrict__ sigma = a.sigma + tr * n;
  uint64_t* __restrict__ word = a.word + tr * n;
  uint32_t* __restrict__ pt = a.pt + tr * n;
  uint32_t* __restrict__ list = a.list + tr * n;
  uint32_t* ctr = a.counters + tr * 4;
  const int32_t* __restrict__ pi = a.pi + tr * a.d;
  const uint32_t* __restrict__ rb = a.rbits + tr * a.W32;
  // whole warps take 32 consecutive positions
  for (int64_t m0 = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); m0 < n;
       m0 += (int64_t)gridDim.x * blockDim.x) {
    const int64_t m = m0 + lane;
    const bool tied = m < n && ((m + 1 < n && prefix_eq(pre, n, K, m, m + 1)) ||
                                (m > 0 && prefix_eq(pre, n, K, m - 1, m)));
    const uint32_t mask = __ballot_sync(0xffffffffu, tied);
    if (!mask) continue;
    uint32_t slot = 0;
    if (lane == 0) slot = atomicAdd(&ctr[0], (uint32_t)__popc(mask));
    slot = __shfl_sync(0xffffffffu, slot, 0) + __popc(mask & lanemask_lt());
    uint32_t p = 0;
    if (tied) {
      p = sigma[m];
      if (p >= (uint64_t)n) p = 0;  // cannot happen for a valid order
      pt[m] = p;
      list[slot] = (uint32_t)m;
      if (WORDS == 0) word[m] = __ldg(pkw + p);
    }
    if (WORDS == 1) {
      for (uint32_t rest = mask; rest; rest &= rest - 1) {
        const int src = __ffs(rest) - 1;
        const uint32_t q = __shfl_sync(0xffffffffu, p, src);
        uint64_t wk;
        tie_top_words<1>(a.planes + (size_t)q * a.W32, pi, rb, K, 1, lane, &wk);
        if (lane == src) word[m] = wk;
      }
    }
  }
}

// inv[pi[i]] = i, sign bit set where permuted axis i is reflected; the whole
// block, which synchronises before the table is used.
__device__ __forceinline__ void tie_inverse(const int32_t* __restrict__ pi, const uint32_t* __restrict__ rb, int d,
                                            int32_t* inv) {
  for (int i = threadIdx.x; i < d; i += blockDim.x) {
    const uint32_t refl = (__ldg(rb + (i >> 5)) >> (i & 31)) & 1u;
    inv[__ldg(pi + i)] = i | (int32_t)(refl << 31);
  }
}

// Y[i] = top Lf bits of permuted, reflected coordinate i of point p, filled
// plane word by plane word (Lf loads per 32 coordinates).
__device__ __forceinline__ void tie_load_row(const uint32_t* __restrict__ planes, int64_t n, int d, int W32, int Lf,
                                             const int32_t* inv, uint32_t p, uint8_t* Y) {
  const uint32_t full = (1u << Lf) - 1u;
  for (int m32 = 0; m32 < W32; ++m32) {
    uint32_t w[HF_MAX_BITS];
#pragma unroll
    for (int l = 0; l < HF_MAX_BITS; ++l) w[l] = l < Lf ? __ldg(planes + ((size_t)l * n + p) * W32 + m32) : 0u;
    const int cn = d - 32 * m32 < 32 ? d - 32 * m32 : 32;
    for (int c = 0; c < cn; ++c) {
      uint32_t v = 0;
#pragma unroll
      for (int l = 0; l < HF_MAX_BITS; ++l)
        if (l < Lf) v = (v << 1) | ((w[l] >> c) & 1u);
      const int32_t i = inv[32 * m32 + c];
      Y[i & 0x7fffffff] = (uint8_t)(i < 0 ? v ^ full : v);
    }
  }
}

// Word K of the listed positions: one thread per member, its coordinates' top
// Lf bits in shared memory (row stride 4 x odd bytes: the lanes of a warp, all
// at the same coordinate, fall in distinct banks). Bound by the transform's
// dependent shared-memory steps.
__global__ void tie_words_kernel(const TieArgs a) {
  extern __shared__ __align__(16) unsigned char smraw[];
  if (*(volatile const int*)a.err) return;
  const int64_t n = a.n;
  const size_t tr = blockIdx.y;
  const uint32_t cnt = a.counters[tr * 4];
  if ((uint64_t)blockIdx.x * blockDim.x >= cnt) return;
  const int d = a.d, Lf = a.Lf;
  int32_t* inv = reinterpret_cast<int32_t*>(smraw);
  uint8_t* Y = smraw + (size_t)d * 4 + (size_t)threadIdx.x * a.stride;
  tie_inverse(a.pi + tr * d, a.rbits + tr * a.W32, d, inv);
  __syncthreads();
  for (uint64_t e = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; e < cnt; e += (uint64_t)gridDim.x * blockDim.x) {
    const uint32_t m = a.list[tr * n + e];
    const uint32_t p = a.pt[tr * n + m];
    tie_load_row(a.planes, n, d, a.W32, Lf, inv, p, Y);
    hf_skilling(Y, d, Lf);
    a.word[tr * n + m] = hf_pack_word(Y, d, Lf, a.K);
  }
}

// First position of the run of equal prefixes that holds m (dir = -1), or the
// last one (dir = +1): galloping probes, then bisection; the prefixes are
// sorted, so equality is monotone.
__device__ __forceinline__ int64_t run_edge(const uint64_t* __restrict__ pre, int64_t n, int K, int64_t m, int dir) {
  int64_t in = m, step = 1, out;  // `in` is inside the run, `out` the nearest known position outside
  for (;;) {
    out = in + dir * step;
    if (out < 0 || out >= n) {
      out = out < 0 ? -1 : n;
      break;
    }
    if (!prefix_eq(pre, n, K, m, out)) break;
    in = out;
    step <<= 1;
  }
  while (out - in > 1 || in - out > 1) {
    const int64_t mid = (in + out) >> 1;
    if (mid >= 0 && mid < n && prefix_eq(pre, n, K, m, mid)) in = mid;
    else out = mid;
  }
  return in;
}

// Trees sorted by the first word's top 64 - sh bits only (sort_plan_kernel):
// their runs of equal top bits are ordered by the rest of the K words, points
// in index order among equals, before anything else looks at the order.
// A warp takes 32 positions: a run that lies within them is ordered right
// there, each lane counting its predecessors by shuffles. The positions of the
// other runs are listed (their points and second words by position), and
// refine_rank counts their predecessors, one thread per position; those runs
// are as long as the plan's price allowed, so there is no cap. The first word
// is fetched again in the final order by gather_prefix_kernel.
__global__ void __launch_bounds__(256) refine_warp_kernel(const TieArgs a) {
  if (*(volatile const int*)a.err) return;
  const size_t tr = blockIdx.y;
  const uint32_t s0 = __ldg(a.skip + tr);
  if (!s0) return;
  const int64_t n = a.n;
  const int K = a.K, sh = (int)(s0 - 8u * (K - 1)) * 8, lane = threadIdx.x & 31;
  const uint64_t* __restrict__ w0 = a.prefix + tr * K * n;
  const uint64_t* __restrict__ pk1 = a.pk + tr * a.K2 * n + n;
  uint32_t* __restrict__ sigma = a.sigma + tr * n;
  for (int64_t m0 = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); m0 < n;
       m0 += (int64_t)gridDim.x * blockDim.x) {
    const int64_t m = m0 + lane;
    const bool in = m < n;
    const uint64_t v0 = in ? __ldg(w0 + m) : 0;
    // tie with the next position, the last lane's against the next warp's first
    uint64_t nx = __shfl_down_sync(0xffffffffu, v0, 1);
    if (lane == 31 && m + 1 < n) nx = __ldg(w0 + m + 1);
    const uint32_t eq = __ballot_sync(0xffffffffu, in && m + 1 < n && (v0 >> sh) == (nx >> sh));
    bool enter = false;  // the first position continues the previous warp's run
    if (lane == 0 && m > 0) enter = (__ldg(w0 + m - 1) >> sh) == (v0 >> sh);
    enter = __shfl_sync(0xffffffffu, enter, 0);
    if (!eq && !enter) continue;
    // run [lo, hi] of this lane: the ties below end at the nearest clear bit
    const uint32_t below = ~eq & ((1u << lane) - 1u);  // lanes that do not tie with their next
    const int lo = below ? 32 - __clz(below) : 0;
    const uint32_t above = ~eq >> lane;
    const int hi = above ? lane + __ffs(above) - 1 : 32;  // 32: past the warp
    const bool cross = (lo == 0 && enter) || hi == 32;
    const bool tied = in && (hi > lo || cross);
    uint32_t p = 0;
    uint64_t v1 = 0;
    if (tied) {
      p = sigma[m];
      if (p >= (uint64_t)n) p = 0;  // cannot happen for a valid order
      if (K > 1) v1 = __ldg(pk1 + p);
    }
    const uint32_t far = __ballot_sync(0xffffffffu, tied && cross);
    if (far) {
      uint32_t slot = 0;
      if (lane == 0) slot = atomicAdd(&a.counters[tr * 4 + 3], (uint32_t)__popc(far));
      slot = __shfl_sync(0xffffffffu, slot, 0) + __popc(far & lanemask_lt());
      if (tied && cross) {
        a.pt[tr * n + m] = p;
        a.list[tr * n + slot] = (uint32_t)m;
        if (K > 1) a.word[tr * n + m] = v1;
      }
    }
    const bool near = tied && !cross;
    const int len = near ? hi - lo + 1 : 1;
    const int most = __reduce_max_sync(0xffffffffu, len);
    int rank = 0, other = lane;
    for (int it = 1; it < most; ++it) {
      other = other == hi ? lo : other + 1;  // around the run
      const int src = near ? other : lane;
      const uint64_t x = __shfl_sync(0xffffffffu, v0, src), y = __shfl_sync(0xffffffffu, v1, src);
      if (it < len && (x < v0 || (x == v0 && (y < v1 || (y == v1 && src < lane))))) ++rank;
    }
    if (near) sigma[m0 + lo + rank] = p;  // every member's point was read above
  }
}

// Edge of the run of equal top bits that holds position m (dir = -1: first,
// +1: last), by galloping probes and bisection.
__device__ __forceinline__ int64_t bits_edge(const uint64_t* __restrict__ w0, int64_t n, int sh, int64_t m, int dir) {
  const uint64_t v = __ldg(w0 + m) >> sh;
  int64_t in = m, step = 1, out;
  for (;;) {
    out = in + dir * step;
    if (out < 0 || out >= n) {
      out = out < 0 ? -1 : n;
      break;
    }
    if ((__ldg(w0 + out) >> sh) != v) break;
    in = out;
    step <<= 1;
  }
  while (out - in > 1 || in - out > 1) {
    const int64_t mid = (in + out) >> 1;
    if (mid >= 0 && mid < n && (__ldg(w0 + mid) >> sh) == v) in = mid;
    else out = mid;
  }
  return in;
}

__global__ void __launch_bounds__(256) refine_rank_kernel(const TieArgs a) {
  if (*(volatile const int*)a.err) return;
  const size_t tr = blockIdx.y;
  const uint32_t s0 = __ldg(a.skip + tr);
  if (!s0) return;
  const int64_t n = a.n;
  const int K = a.K, sh = (int)(s0 - 8u * (K - 1)) * 8;
  const uint64_t* __restrict__ w0 = a.prefix + tr * K * n;
  const uint64_t* __restrict__ w1 = a.word + tr * n;
  const uint32_t cnt = a.counters[tr * 4 + 3];
  for (uint64_t e = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; e < cnt; e += (uint64_t)gridDim.x * blockDim.x) {
    const int64_t m = a.list[tr * n + e];
    const int64_t lo = bits_edge(w0, n, sh, m, -1), hi = bits_edge(w0, n, sh, m, 1);
    const uint64_t v0 = __ldg(w0 + m), v1 = K > 1 ? w1[m] : 0;
    uint32_t below = 0;
    if (sh == 0) {  // the first words are equal throughout
      for (int64_t g = lo; g <= hi; ++g) {
        const uint64_t y = K > 1 ? w1[g] : 0;
        below += (y < v1 || (y == v1 && g < m)) ? 1u : 0u;
      }
    } else {
      for (int64_t g = lo; g <= hi; ++g) {
        const uint64_t x = __ldg(w0 + g);
        if (x < v0) {
          ++below;
        } else if (x == v0) {
          const uint64_t y = K > 1 ? w1[g] : 0;
          below += (y < v1 || (y == v1 && g < m)) ? 1u : 0u;
        }
      }
    }
    a.sigma[tr * n + lo + below] = a.pt[tr * n + m];
  }
}

// One thread per listed position. The run's words are read in order (the
// lanes of a warp mostly share a run: broadcast loads). Ties on every word at
// hand (word K, and words K+1 .. K2-1 when the key kernel formed them) stay in
// index order, which is position order; the first of a tied group lists the
// group as a sub-run when the key has more words.
__global__ void __launch_bounds__(256) tie_rank_kernel(const TieArgs a) {
  if (*(volatile const int*)a.err) return;
  const int64_t n = a.n;
  const size_t tr = blockIdx.y;
  uint32_t* ctr = a.counters + tr * 4;
  const uint32_t cnt = ctr[0];
  const int K = a.K;
  const uint64_t* __restrict__ pre = a.prefix + tr * K * n;
  const uint64_t* __restrict__ pk = a.pk + tr * a.K2 * n;
  const uint64_t* __restrict__ word = a.word + tr * n;
  const uint32_t* __restrict__ pt = a.pt + tr * n;
  uint32_t* __restrict__ sigma = a.sigma + tr * n;
  uint2* big = a.big + tr * a.big_cap;
  const int known = a.K2 > K + 1 ? a.K2 : K + 1;  // key words at hand
  for (uint64_t e = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; e < cnt; e += (uint64_t)gridDim.x * blockDim.x) {
    const int64_t m = a.list[tr * n + e];
    const int64_t lo = run_edge(pre, n, K, m, -1), hi = run_edge(pre, n, K, m, 1);
    if (hi - lo >= TIE_RUN_CAP) {
      if (m == lo) {
        const uint32_t r = atomicAdd(&ctr[1], 1u);
        if (r < a.big_cap) big[r] = make_uint2((uint32_t)lo, (uint32_t)(hi - lo + 1));
      }
      continue;
    }
    const uint64_t own = word[m];
    const uint32_t p = pt[m];
    uint32_t rank = 0, before = 0, after = 0;
    for (int64_t g = lo; g <= hi; ++g) {
      const uint64_t v = word[g];
      if (v < own) ++rank;
      if (v == own && g != m) {
        int c = 0;
        for (int w = K + 1; w < a.K2 && c == 0; ++w) {
          const uint64_t x = __ldg(pk + (size_t)w * n + pt[g]), y = __ldg(pk + (size_t)w * n + p);
          c = x < y ? -1 : (x > y ? 1 : 0);
        }
        if (c < 0) ++rank;
        else if (c == 0 && g < m) ++before;
        else if (c == 0) ++after;
      }
    }
    sigma[lo + rank + before] = p;
    if (known < a.W && before == 0 && after > 0) {
      const uint2 sub = make_uint2((uint32_t)(lo + rank), after + 1);
      if ((int)after < tie_hard_cap(a.W)) {
        a.hard[tr * n + atomicAdd(&ctr[2], 1u)] = sub;
      } else {
        const uint32_t r = atomicAdd(&ctr[1], 1u);
        if (r < a.big_cap) big[r] = sub;
      }
    }
  }
}

// -1 / 0 / +1 comparing the N words x and y.
template <int N>
__device__ __forceinline__ int cmp_words(const uint64_t (&x)[N], const uint64_t (&y)[N]) {
  int c = 0;
#pragma unroll
  for (int i = N - 1; i >= 0; --i) c = x[i] < y[i] ? -1 : (x[i] > y[i] ? 1 : c);
  return c;
}

// Sub-runs that tie on every word at hand, ranked by the next words of the top
// bit level where there are any (a.top), and if some members tie on those too,
// by (full key, index) from full keys in the block's slice of global scratch.
// Sub-runs of few members (a warp's share of the block's rows) take a warp each,
// eight at a time in a block, the others the whole block, one member per thread.
// A member's full key is a serial chain of one thread, 60 us at d = 384, however
// many lanes run beside it; its top-level words take a warp about 1 us. Near-
// duplicates make sub-runs by the hundred thousand. Builds of 500,000 x 384, T =
// 4, groups of 10 copies with 5 % / 1 % / 0.1 % noise: 2.5 / 40.2 / 32.8 ms; with
// one block per sub-run and full keys at once 39.4 / 198 / 130; with one block
// per run of equal prefixes, four words and then full keys for the whole run,
// 9.6 / 287 / 294. 50,000 x 768, T = 1, in groups of 1,000 with 20 % noise, where
// the few sub-runs' chain is a third of the build: 0.755 -> 0.45 ms.
__global__ void __launch_bounds__(TIE_HARD_WARPS * 32) tie_hard_kernel(const TieArgs a,
                                                                       uint64_t* __restrict__ fk_scratch) {
  extern __shared__ __align__(16) unsigned char smraw[];
  if (*(volatile const int*)a.err) return;
  const int64_t n = a.n;
  const int d = a.d, W = a.W, top = a.top, cap = tie_hard_cap(W);
  const bool all = a.K + 1 + top >= W;  // the key has no words beyond those
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int share = a.rows / TIE_HARD_WARPS;  // members of a warp's sub-run, 32 at most
  uint64_t* tw = reinterpret_cast<uint64_t*>(smraw);                        // [cap][TIE_TOP_WORDS]
  uint32_t* pt = reinterpret_cast<uint32_t*>(tw + (size_t)cap * TIE_TOP_WORDS);  // [cap]
  int32_t* inv = reinterpret_cast<int32_t*>(pt + cap);                      // [d]
  uint8_t* Y = reinterpret_cast<uint8_t*>(inv + d);                         // [rows][stride]
  uint64_t* fk = fk_scratch + (size_t)blockIdx.x * cap * W;
  auto full_key = [&](uint32_t p, int row, uint64_t* out) {
    uint8_t* y = Y + (size_t)row * a.stride;
    tie_load_row(a.planes, n, d, a.W32, a.bits, inv, p, y);
    hf_skilling(y, d, a.bits);
    for (int w = 0; w < W; ++w) out[w] = hf_pack_word(y, d, a.bits, w);
  };
  for (int tr = 0; tr < a.tb; ++tr) {
    const uint32_t nruns = a.counters[(size_t)tr * 4 + 2];
    uint32_t* sigma = a.sigma + (size_t)tr * n;
    const uint2* hard = a.hard + (size_t)tr * n;
    const int32_t* pi = a.pi + (size_t)tr * d;
    const uint32_t* rb = a.rbits + (size_t)tr * a.W32;
    // trees start at different blocks, so that a few sub-runs per tree spread
    const uint32_t first = (blockIdx.x + (uint32_t)tr * 37u) % gridDim.x;
    if (first >= nruns) continue;
    tie_inverse(pi, rb, d, inv);
    __syncthreads();
    // short sub-runs, a warp each
    for (uint64_t r = first + (uint64_t)warp * gridDim.x; r < nruns; r += (uint64_t)TIE_HARD_WARPS * gridDim.x) {
      const uint2 run = hard[r];
      const int len = (int)run.y;
      if (len > share) continue;
      const bool in = lane < len;
      uint32_t p = in ? sigma[run.x + lane] : 0;
      if (p >= (uint64_t)n) p = 0;  // cannot happen for a valid order
      uint64_t own[TIE_TOP_WORDS] = {};
      for (int e = 0; e < len && top; ++e) {
        uint64_t w[TIE_TOP_WORDS];
        tie_top_words<TIE_TOP_WORDS>(a.planes + (size_t)__shfl_sync(0xffffffffu, p, e) * a.W32, pi, rb, a.K + 1, top,
                                     lane, w);
#pragma unroll
        for (int i = 0; i < TIE_TOP_WORDS; ++i)
          if (lane == e) own[i] = w[i];
      }
      // members that tie on those stay in position order, which is index order
      int rank = 0;
      bool tie = false;
      for (int g = 0; g < len; ++g) {
        uint64_t o[TIE_TOP_WORDS];
#pragma unroll
        for (int i = 0; i < TIE_TOP_WORDS; ++i) o[i] = __shfl_sync(0xffffffffu, own[i], g);
        const int c = cmp_words(o, own);
        rank += c < 0 || (c == 0 && g < lane) ? 1 : 0;
        tie |= in && c == 0 && g != lane;
      }
      if (!all && __any_sync(0xffffffffu, tie)) {
        uint64_t* wk = fk + (size_t)(warp * share) * W;
        if (in) full_key(p, warp * share + lane, wk + (size_t)lane * W);
        __syncwarp();
        rank = 0;
        for (int g = 0; g < len; ++g) {
          const uint32_t pg = __shfl_sync(0xffffffffu, p, g);
          if (in) rank += full_less(wk + (size_t)g * W, pg, wk + (size_t)lane * W, p, W) ? 1 : 0;
        }
        __syncwarp();  // the keys are read before the warp's next sub-run
      }
      if (in) sigma[run.x + rank] = p;
    }
    __syncthreads();  // the rows and the scratch change hands
    // the others, the whole block each (len <= cap <= the block's threads)
    for (uint64_t r = first; r < nruns; r += gridDim.x) {
      const uint2 run = hard[r];
      const int len = (int)run.y;
      if (len <= share) continue;
      const bool in = tid < len;
      uint32_t p = in ? sigma[run.x + tid] : 0;
      if (p >= (uint64_t)n) p = 0;  // cannot happen for a valid order
      if (in) pt[tid] = p;
      __syncthreads();
      for (int e = warp; e < len && top; e += TIE_HARD_WARPS) {
        uint64_t w[TIE_TOP_WORDS];
        tie_top_words<TIE_TOP_WORDS>(a.planes + (size_t)pt[e] * a.W32, pi, rb, a.K + 1, top, lane, w);
        if (lane == 0)
#pragma unroll
          for (int i = 0; i < TIE_TOP_WORDS; ++i) tw[e * TIE_TOP_WORDS + i] = w[i];
      }
      __syncthreads();
      int rank = 0;
      bool tie = false;
      if (in && top) {
        uint64_t own[TIE_TOP_WORDS], o[TIE_TOP_WORDS];
#pragma unroll
        for (int i = 0; i < TIE_TOP_WORDS; ++i) own[i] = tw[tid * TIE_TOP_WORDS + i];
        for (int g = 0; g < len; ++g) {
#pragma unroll
          for (int i = 0; i < TIE_TOP_WORDS; ++i) o[i] = tw[g * TIE_TOP_WORDS + i];
          const int c = cmp_words(o, own);
          rank += c < 0 || (c == 0 && g < tid) ? 1 : 0;
          tie |= c == 0 && g != tid;
        }
      } else {
        rank = tid;
        tie = in;
      }
      if (!all && __syncthreads_or(tie)) {
        if (tid < a.rows)
          for (int e = tid; e < len; e += a.rows) full_key(pt[e], tid, fk + (size_t)e * W);
        __syncthreads();
        rank = 0;
        if (in)
          for (int g = 0; g < len; ++g)
            rank += full_less(fk + (size_t)g * W, pt[g], fk + (size_t)tid * W, p, W) ? 1 : 0;
      }
      if (in) sigma[run.x + rank] = p;
      __syncthreads();  // pt, tw and the keys are read before the next sub-run
    }
    __syncthreads();  // the table is read before the next tree's
  }
}

// Big runs: full keys into global scratch, then a bitonic network over all
// big-run elements of one tree ordered by (run, full key, point).
__global__ void big_fill_kernel(const uint32_t* __restrict__ planes, int64_t n, int d, int W32,
                                int bits, int W, const int32_t* __restrict__ pi,
                                const uint32_t* __restrict__ rbits, const uint2* __restrict__ big,
                                const uint32_t* __restrict__ offs, int nbig,
                                const uint32_t* __restrict__ sigma, uint64_t* __restrict__ fk,
                                uint32_t* __restrict__ item_pt, uint32_t* __restrict__ item_run,
                                uint8_t* __restrict__ yscratch) {
  const int r = blockIdx.x;
  if (r >= nbig) return;
  const uint2 run = big[r];
  uint8_t* y = yscratch + ((size_t)blockIdx.x * blockDim.x + threadIdx.x) * d;
  for (uint32_t e = threadIdx.x; e < run.y; e += blockDim.x) {
    const uint32_t slot = offs[r] + e;
    const uint32_t p = sigma[run.x + e];
    item_pt[slot] = p;
    item_run[slot] = (uint32_t)r;
    hf_load_coords_planes(planes, n, d, W32, bits, pi, rbits, p, y);
    hf_skilling(y, d, bits);
    for (int w = 0; w < W; ++w) fk[(size_t)slot * W + w] = hf_pack_word(y, d, bits, w);
  }
}

__device__ __forceinline__ bool item_less(uint32_t a, uint32_t b, const uint64_t* fk,
                                          const uint32_t* pt, const uint32_t* rn, int W,
                                          uint32_t total) {
  const bool va = a < total, vb = b < total;
  if (va != vb) return va;  // padding sorts last
  if (!va) return false;
  if (rn[a] != rn[b]) return rn[a] < rn[b];
  return full_less(fk + (size_t)a * W, pt[a], fk + (size_t)b * W, pt[b], W);
}

__global__ void bitonic_step_kernel(uint32_t* __restrict__ ord, uint32_t m, uint32_t j, uint32_t kk,
                                    const uint64_t* __restrict__ fk, const uint32_t* __restrict__ pt,
                                    const uint32_t* __restrict__ rn, int W, uint32_t total) {
  const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= m) return;
  const uint32_t l = i ^ j;
  if (l <= i) return;
  const uint32_t a = ord[i], b = ord[l];
  const bool up = (i & kk) == 0;
  const bool sw = up ? item_less(b, a, fk, pt, rn, W, total) : item_less(a, b, fk, pt, rn, W, total);
  if (sw) {
    ord[i] = b;
    ord[l] = a;
  }
}

__global__ void big_write_kernel(const uint32_t* __restrict__ ord, uint32_t total,
                                 const uint32_t* __restrict__ pt, const uint32_t* __restrict__ rn,
                                 const uint2* __restrict__ big, const uint32_t* __restrict__ offs,
                                 uint32_t* __restrict__ sigma) {
  const uint32_t s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= total) return;
  const uint32_t it = ord[s];
  const uint32_t r = rn[it];
  sigma[big[r].x + (s - offs[r])] = pt[it];
}

__global__ void iota_kernel(uint32_t* a, uint32_t m) {
  const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < m) a[i] = i;
}

constexpr int TIE_BLOCKS = 152 * 2;

// Shared memory of a tie_hard block, and its coordinate rows (d bytes each): as
// many as let two blocks share an SM, 32 at least (131 KB at d = 4096).
size_t tie_hard_smem(int W, int d, int stride, int rows) {
  return (size_t)tie_hard_cap(W) * (TIE_TOP_WORDS * 8 + 4) + (size_t)d * 4 + (size_t)rows * stride;
}
int tie_hard_rows(int W, int d, int stride) {
  int rows = tie_hard_cap(W);
  while (rows > 32 && tie_hard_smem(W, d, stride, rows) > 112 * 1024) rows >>= 1;
  return rows;
}

// Levels that word K needs, and the row stride of tie_words.
int tie_levels(int d, int bits, int K) {
  const int64_t lf = ((int64_t)64 * (K + 1) + d - 1) / d;
  return (int)(lf < bits ? lf : bits);
}

}  // namespace

static cudaError_t set_attr(const void* fn, size_t bytes) {
  return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

// Sorts trees t0 .. t0 + tb - 1 (their key words are at f->pk, tree j of the
// batch at f->pk + j * K2 * n) into f->prefix / f->sigma, then fixes each
// tree's runs of equal prefixes.
int sort_batch(hf_forest* f, int t0, int tb, cudaStream_t s) {
  const int64_t n = f->n;
  const int K = f->K, K2 = f->K2;
  const int64_t ntiles = (n + TILE - 1) / TILE;
  const int passes = 8 * K;
  const size_t per_pass = (size_t)tb * (ntiles + 1) * 256 + 1;  // status rows (+ spare row per tree) + ticket
  const int64_t pk_ts = (int64_t)K2 * n;
  const int64_t hist_ts = (int64_t)K * 8 * 256;
  uint32_t* status = f->sort.status;

  // the plan's words, the histograms and the look-back words are one run
  cudaMemsetAsync(f->sort.skip, 0,
                  (size_t)(status - f->sort.skip) * sizeof(uint32_t) + per_pass * passes * sizeof(uint32_t), s);
  const size_t hsm = (size_t)hist_ts * sizeof(uint32_t);
  set_attr((const void*)digit_hist_kernel, hsm);
  digit_hist_kernel<<<dim3(hf_blocks(n, 512, 152 * 8 / tb + 1), (unsigned)tb), 512, hsm, s>>>(f->pk, pk_ts, n, K,
                                                                                            f->sort.hist);
  hf_after_launch("digit_hist_kernel", s);
  hist_scan_kernel<<<(unsigned)(tb * K * 8), 256, 0, s>>>(f->sort.hist);
  hf_after_launch("hist_scan_kernel", s);

  const size_t psm = sizeof(PassSmem);
  set_attr((const void*)onesweep_kernel<false>, psm);
  set_attr((const void*)onesweep_kernel<true>, psm);

  // first pass of each tree: the plan handles one or two words; the stall test
  // needs its first pass
  uint32_t* skip = f->sort.skip;
  if (K <= 2 && !f->test_stall) {
    if (n >= PLAN_LARGE)
      sort_plan_kernel<4096><<<(unsigned)tb, 1024, 0, s>>>(f->pk, pk_ts, n, K, tb, skip, f->sort.first + t0);
    else
      sort_plan_kernel<1024><<<(unsigned)tb, 1024, 0, s>>>(f->pk, pk_ts, n, K, tb, skip, f->sort.first + t0);
    hf_after_launch("sort_plan_kernel", s);
  }

  PassArgs a{};
  a.skip = skip;
  a.err = f->err;
  a.n = n;
  a.ntiles = ntiles;
  a.spin_ns = (uint64_t)f->spin_limit_us * 1000ull;
  a.TB = tb;
  a.goff_ts = hist_ts;
  a.gather_src_ts = pk_ts;
  const unsigned grid = (unsigned)(ntiles * tb);
  int pass = 0;
  for (int w = K - 1; w >= 0; --w) {
    for (int b = 0; b < 8; ++b, ++pass) {
      const bool gather = (w < K - 1) && b == 0;
      const bool last = pass == passes - 1;
      a.pass = (uint32_t)pass;
      a.first_src = f->pk + (size_t)w * n;
      a.first_src_ts = pk_ts;
      a.gather_src = gather ? f->pk + (size_t)w * n : nullptr;
      if (last) {
        a.keys_out = f->prefix + (size_t)t0 * K * n;  // word 0 of each tree's prefix
        a.keys_out_ts = (int64_t)K * n;
        a.vals_out = f->sigma + (size_t)t0 * n;
        a.vals_out_ts = n;
      } else {
        a.keys_out = (pass & 1) ? f->sort.keys_b : f->sort.keys_a;
        a.keys_out_ts = n;
        a.vals_out = (pass & 1) ? f->sort.vals_b : f->sort.vals_a;
        a.vals_out_ts = n;
      }
      a.goff = f->sort.hist + (size_t)(w * 8 + b) * 256;
      a.status = status + per_pass * pass;
      a.ticket = a.status + (size_t)tb * (ntiles + 1) * 256;
      a.shift = 8 * b;
      a.stall = (f->test_stall && pass == 0) ? 1 : 0;
      if (gather)
        onesweep_kernel<true><<<grid, NT, psm, s>>>(a);
      else
        onesweep_kernel<false><<<grid, NT, psm, s>>>(a);
      hf_after_launch("onesweep_kernel", s);
      a.keys_in = a.keys_out;
      a.keys_in_ts = a.keys_out_ts;
      a.vals_in = a.vals_out;
      a.vals_in_ts = a.vals_out_ts;
    }
  }
  // per tree blocks of the launches below: about 16 blocks per SM over all trees
  const int64_t tree_cap = (152 * 16 + tb - 1) / tb;
  const dim3 grid16(hf_blocks(n, 256, tree_cap), (unsigned)tb);
  {
    TieArgs a{};
    a.skip = skip;
    a.prefix = f->prefix + (size_t)t0 * K * n;
    a.pk = f->pk;
    a.sigma = f->sigma + (size_t)t0 * n;
    a.word = f->sort.keys_a;
    a.hard = reinterpret_cast<uint2*>(f->sort.keys_b);
    a.pt = f->sort.vals_a;
    a.list = f->sort.vals_b;
    a.big = f->tie.big_runs + (size_t)t0 * f->tie.big_cap;
    a.counters = f->tie.counters + (size_t)t0 * 4;
    a.planes = f->planes;
    a.pi = f->pi + (size_t)t0 * f->d;
    a.rbits = f->rbits + (size_t)t0 * f->W32;
    a.err = f->err;
    a.n = n;
    a.big_cap = f->tie.big_cap;
    a.d = f->d;
    a.W32 = f->W32;
    a.bits = f->bits;
    a.W = f->W;
    a.K = K;
    a.K2 = K2;
    a.Lf = tie_levels(f->d, f->bits, K);
    a.tb = tb;
    a.stride = ((f->d + 3) / 4 | 1) * 4;
    if (K <= 2) {
      refine_warp_kernel<<<grid16, 256, 0, s>>>(a);
      hf_after_launch("refine_warp_kernel", s);
      refine_rank_kernel<<<grid16, 256, 0, s>>>(a);
      hf_after_launch("refine_rank_kernel", s);
    }
    gather_prefix_kernel<<<grid16, 256, 0, s>>>(f->pk, pk_ts, f->sigma + (size_t)t0 * n, n, K, skip,
                                               f->prefix + (size_t)t0 * K * n, f->err);
    hf_after_launch("gather_prefix_kernel", s);
    // Equal prefixes, settled on the device right away. With K == W the prefix
    // is the whole key: equal prefixes are equal keys, already in index order.
    if (K >= f->W) return cudaGetLastError() == cudaSuccess ? HF_OK : HF_ECUDA;
    const dim3 grid = grid16;
    if (K2 > K) {
      tie_mark_kernel<0><<<grid, 256, 0, s>>>(a);
      hf_after_launch("tie_mark_kernel", s);
    } else if (f->d >= 64 * (K + 1)) {
      tie_mark_kernel<1><<<grid, 256, 0, s>>>(a);
      hf_after_launch("tie_mark_kernel", s);
    } else {
      tie_mark_kernel<2><<<grid, 256, 0, s>>>(a);
      hf_after_launch("tie_mark_kernel", s);
      // d < 64 (K + 1) <= 576 here: a block of 128 rows holds 75 KB at most
      const size_t sm = (size_t)f->d * 4 + (size_t)128 * a.stride;
      set_attr((const void*)tie_words_kernel, sm);
      tie_words_kernel<<<dim3(hf_blocks(n, 128, 2 * tree_cap), (unsigned)tb), 128, sm, s>>>(a);
      hf_after_launch("tie_words_kernel", s);
    }
    tie_rank_kernel<<<grid, 256, 0, s>>>(a);
    hf_after_launch("tie_rank_kernel", s);
    if ((K2 > K + 1 ? K2 : K + 1) < f->W) {
      a.rows = tie_hard_rows(f->W, f->d, a.stride);
      if (K2 == K && f->d >= 64 * (K + 1)) a.top = std::min(TIE_TOP_WORDS, f->d / 64 - (K + 1));
      const size_t sm = tie_hard_smem(f->W, f->d, a.stride, a.rows);
      set_attr((const void*)tie_hard_kernel, sm);
      tie_hard_kernel<<<TIE_BLOCKS, TIE_HARD_WARPS * 32, sm, s>>>(a, f->tie.fk);
      hf_after_launch("tie_hard_kernel", s);
    }
  }
  return cudaGetLastError() == cudaSuccess ? HF_OK : HF_ECUDA;
}

// Segmented forest: one more stable LSD pass per tree, keyed by the set of
// each point (the most significant digit of the order), gathered through the
// current order. Equal sets keep their relative order, so every set's points
// stay in their own Hilbert order and set s occupies positions off[s] ..
// off[s+1]-1. Up to 256 sets (one 8-bit digit).
int segment_pass(hf_forest* f, const uint64_t* seg64, cudaStream_t s) {
  const int64_t n = f->n;
  const int nseg = f->nseg;
  if (nseg < 2 || nseg > 256) return HF_EINVAL;
  const int64_t ntiles = (n + TILE - 1) / TILE;
  std::vector<uint32_t> goff(256, (uint32_t)n);
  for (int g = 0; g < nseg; ++g) goff[g] = (uint32_t)f->seg_off_h[g];
  if (cudaMemcpyAsync(f->sort.hist, goff.data(), 256 * sizeof(uint32_t), cudaMemcpyHostToDevice, s) != cudaSuccess)
    return HF_ECUDA;
  const size_t psm = sizeof(PassSmem);
  set_attr((const void*)onesweep_kernel<true>, psm);
  for (int t0 = 0; t0 < f->T; t0 += f->TB) {
    const int tb = f->T - t0 < f->TB ? f->T - t0 : f->TB;
    const size_t words = (size_t)tb * (ntiles + 1) * 256 + 1;
    cudaMemsetAsync(f->sort.status, 0, words * sizeof(uint32_t), s);
    PassArgs a{};
    a.err = f->err;
    a.n = n;
    a.ntiles = ntiles;
    a.spin_ns = (uint64_t)f->spin_limit_us * 1000ull;
    a.TB = tb;
    a.vals_in = f->sigma + (size_t)t0 * n;
    a.vals_in_ts = n;
    a.gather_src = seg64;
    a.gather_src_ts = 0;
    a.keys_out = f->sort.keys_a;
    a.keys_out_ts = n;
    a.vals_out = f->sort.vals_a;
    a.vals_out_ts = n;
    a.goff = f->sort.hist;
    a.goff_ts = 0;
    a.status = f->sort.status;
    a.ticket = f->sort.status + (size_t)tb * (ntiles + 1) * 256;
    a.shift = 0;
    onesweep_kernel<true><<<(unsigned)(ntiles * tb), NT, psm, s>>>(a);
    hf_after_launch("onesweep_kernel<segment>", s);
    cudaMemcpyAsync(f->sigma + (size_t)t0 * n, f->sort.vals_a, (size_t)tb * n * sizeof(uint32_t),
                    cudaMemcpyDeviceToDevice, s);
  }
  return cudaGetLastError() == cudaSuccess ? HF_OK : HF_ECUDA;
}

// Host side of the big-run path; called after the build's sync, when the
// host knows how many big runs tree t has.
int tie_fixup_big(hf_forest* f, int t, uint32_t nbig, cudaStream_t s) {
  if (nbig == 0) return HF_OK;
  if (nbig > f->tie.big_cap) return HF_ECUDA;
  const int64_t n = f->n;
  std::vector<uint2> runs(nbig);
  if (cudaMemcpy(runs.data(), f->tie.big_runs + (size_t)t * f->tie.big_cap, nbig * sizeof(uint2),
                 cudaMemcpyDeviceToHost) != cudaSuccess)
    return HF_ECUDA;
  std::vector<uint32_t> offs(nbig);
  uint64_t total = 0;
  for (uint32_t r = 0; r < nbig; ++r) {
    offs[r] = (uint32_t)total;
    total += runs[r].y;
  }
  uint32_t m = 1;
  while (m < total) m <<= 1;
  const int W = f->W;
  const int tt = 64;
  uint64_t* fk = nullptr;
  uint32_t *pt = nullptr, *rn = nullptr, *ord = nullptr, *doffs = nullptr;
  uint8_t* ys = nullptr;
  uint2* druns = f->tie.big_runs + (size_t)t * f->tie.big_cap;
  int rc = HF_OK;
  auto take = [&](void** p, size_t bytes) {
    if (rc == HF_OK && hf_dalloc_bytes(p, bytes, s) != cudaSuccess) {
      cudaGetLastError();
      rc = HF_ENOMEM;
    }
  };
  take((void**)&fk, (size_t)total * W * 8);
  take((void**)&pt, total * 4);
  take((void**)&rn, total * 4);
  take((void**)&ord, (size_t)m * 4);
  take((void**)&doffs, nbig * 4);
  take((void**)&ys, (size_t)nbig * tt * f->d);
  if (rc == HF_OK) {
    cudaMemcpyAsync(doffs, offs.data(), nbig * 4, cudaMemcpyHostToDevice, s);
    uint32_t* sig = f->sigma + (size_t)t * n;
    big_fill_kernel<<<nbig, tt, 0, s>>>(f->planes, n, f->d, f->W32, f->bits, W, f->pi + (size_t)t * f->d,
                                        f->rbits + (size_t)t * f->W32, druns, doffs, (int)nbig, sig, fk, pt,
                                        rn, ys);
    hf_after_launch("big_fill_kernel", s);
    iota_kernel<<<hf_blocks(m, 256), 256, 0, s>>>(ord, m);
    hf_after_launch("iota_kernel", s);
    for (uint32_t kk = 2; kk <= m; kk <<= 1)
      for (uint32_t j = kk >> 1; j > 0; j >>= 1) {
        bitonic_step_kernel<<<hf_blocks(m, 256), 256, 0, s>>>(ord, m, j, kk, fk, pt, rn, W, (uint32_t)total);
        hf_after_launch("bitonic_step_kernel", s);
      }
    big_write_kernel<<<hf_blocks(total, 256), 256, 0, s>>>(ord, (uint32_t)total, pt, rn, druns, doffs, sig);
    hf_after_launch("big_write_kernel", s);
  }
  // stream-ordered frees: the pool hands the memory to the next user of s
  // without a device-wide synchronisation
  hf_dfree_bytes(fk, s);
  hf_dfree_bytes(pt, s);
  hf_dfree_bytes(rn, s);
  hf_dfree_bytes(ord, s);
  hf_dfree_bytes(doffs, s);
  hf_dfree_bytes(ys, s);
  if (rc == HF_OK && cudaGetLastError() != cudaSuccess) rc = HF_ECUDA;
  return rc;
}

// Words of the sub-runs' full-key scratch.
size_t tie_scratch_words(int W) { return (size_t)TIE_BLOCKS * tie_hard_cap(W) * W; }

// Launches of the fix-up per batch (sort_batch's own conditions).
int tie_launches(const hf_forest* f) {
  if (f->K >= f->W) return 0;
  const bool words = f->K2 == f->K && f->d < 64 * (f->K + 1);
  const bool hard = (f->K2 > f->K + 1 ? f->K2 : f->K + 1) < f->W;
  return 2 + (words ? 1 : 0) + (hard ? 1 : 0);
}

// Runs and sub-runs on the big list are longer than this.
int tie_big_min(int W) { return tie_hard_cap(W); }

size_t sort_status_words(int64_t n, int K, int tb) {
  const int64_t ntiles = (n + TILE - 1) / TILE;
  return ((size_t)tb * (ntiles + 1) * 256 + 1) * 8 * K;
}
