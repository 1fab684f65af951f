// Batched query search.
//
// Paper, Section 2: since the Hilbert order is a total order, binary search
// locates an arbitrary point in a sorted set; Algorithm 1 then takes the
// candidates near each query's position in every tree and keeps the top k by
// vector distance. The paper simulates a collective Hilbert sort of all queries
// on the CPU; here every query is located independently, which parallelises
// trivially.
//
// One warp per query, looping over the trees; the query's top-k list lives in
// registers across the warp (entry e in lane e % 32, slot e / 32).
//  * Key prefix: when the first K key words lie in the top bit level (d >=
//    64K) the warp forms them with ballots (running XOR of the permuted,
//    reflected top bits); otherwise lane 0 runs the transform.
//  * Locate: 32-way probing rounds find the lower bound among the sorted
//    prefixes; only when the prefix at that position equals the query's does
//    a second search find the end of the equal run, inside which lane 0
//    refines the position by full keys (computed on demand from the planes).
//  * Score: the window's candidates go 32 at a time. Every lane reads its 4
//    coordinates of each candidate row (a row is read by the warp in 512-byte
//    coalesced pieces) and keeps one partial sum per candidate; a transposing
//    butterfly (31 shuffles) leaves candidate j's distance in lane j. The
//    butterfly adds lane partials in the same tree for every candidate, so a
//    (query, point) pair gets the same value in every tree.
//  * Merge: the 32 scored candidates are sorted across the warp and inserted
//    in ascending order until the first one that cannot enter.
//  * Large batches locate their queries in a launch of their own and read a
//    half-width copy of the points first (search16_kernel): the distance to a
//    point's BF16 copy, less the copy's distance from the point, bounds the
//    point's distance from below, and only candidates whose bound does not
//    exceed the list's last entry are scored, from the float32 rows and in the
//    arithmetic above. The lists are the same. 10,000 queries, 3M x 384, T = 64,
//    w = 50 (98 GB of float32 rows): 18.2 -> 11.1 ms, 12.3 with the copy's
//    making; bound by the screen's instructions (about 12 per row and four
//    coordinates), no longer by HBM.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math.h>

#include <type_traits>

#include "hf_internal.cuh"
#include "hilbert_device.cuh"

namespace {

constexpr int SWARPS = 4;
constexpr unsigned FULL = 0xffffffffu;

// Shared bytes per warp: query prefix (K words), candidate ids (32 words),
// two coordinate scratch rows (d bytes each), rounded to 16.
__host__ __device__ __forceinline__ size_t search_per_warp(int K, int d) {
  return ((size_t)K * 8 + 32 * 4 + 2 * (size_t)d + 15) & ~(size_t)15;
}

__device__ __forceinline__ bool lessp(float da, uint32_t ia, float db, uint32_t ib) {
  return da < db || (da == db && ia < ib);
}

// -1 / 0 / +1 comparing the sorted prefix at position m with the query prefix.
__device__ __forceinline__ int cmp_prefix(const uint64_t* __restrict__ pre, int64_t n, int K, int64_t m,
                                          const uint64_t* qp) {
  for (int w = 0; w < K; ++w) {
    const uint64_t a = __ldg(pre + (size_t)w * n + m);
    if (a != qp[w]) return a < qp[w] ? -1 : 1;
  }
  return 0;
}

// Full-key comparison: is the key of transformed Yd smaller than that of Yq?
__device__ __forceinline__ bool full_key_less(const uint8_t* Yd, const uint8_t* Yq, int d, int bits, int W) {
  for (int w = 0; w < W; ++w) {
    const uint64_t a = hf_pack_word(Yd, d, bits, w), b = hf_pack_word(Yq, d, bits, w);
    if (a != b) return a < b;
  }
  return false;
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

struct SearchArgs {
  const float* x;
  int64_t n;
  int d, bits, K, L, W, W32, T;
  const uint32_t* planes;
  const int32_t* pi;
  const uint32_t* rbits;
  const uint64_t* prefix;
  const uint32_t* sigma;
  const float* q;
  const uint8_t* qcodes;
  int64_t nq;
  int k, w;
  uint32_t* out_idx;
  float* out_dist;
  int64_t* out_pos;  // locate_kernel: positions, of one tree [nq] or of all [T][nq]
  int only_tree;     // locate_kernel: that tree, or -1 for all
  int vec4;  // d % 4 == 0 and both matrices 16-byte aligned
  int top;   // the K prefix words lie in the top bit level (d >= 64K)
  // search16_kernel: positions [T][nq], the points in BF16 (row pitch dp) and an
  // upper bound of each one's distance from its copy
  const int64_t* pos;
  const __nv_bfloat16* x16;
  const float* r16;
  int dp;
  // parts of a query: warp `part` takes trees tp, tp + tsplit, ... and, in
  // each window, the 32-candidate chunks cp, cp + csplit, ... (part = tp *
  // csplit + cp). One part: out_idx / out_dist hold the result. More: they
  // hold a list of k per part, which merge_parts_kernel merges.
  int tsplit, csplit;
};

// Query prefix from the top bits, the warp taking 32 coordinates per ballot:
// key bit i (i < 64K) is the XOR of the permuted, reflected top bits of
// coordinates 0..i; word w holds bits 64w .. 64w+63, most significant first.
__device__ __forceinline__ void warp_top_prefix(const uint8_t* __restrict__ qc, int bits, int K,
                                                const int32_t* __restrict__ pi, const uint32_t* __restrict__ rb,
                                                uint64_t* qp, int lane) {
  uint32_t carry = 0;
  for (int w = 0; w < K; ++w) {
    uint32_t half[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int i = w * 64 + h * 32 + lane;
      const uint32_t bit = (((uint32_t)qc[__ldg(pi + i)] >> (bits - 1)) ^ (__ldg(rb + (i >> 5)) >> lane)) & 1u;
      uint32_t v = xor_scan_msb(__brev(__ballot_sync(FULL, bit)));
      if (carry) v = ~v;
      carry = v & 1u;
      half[h] = v;
    }
    if (lane == 0) qp[w] = ((uint64_t)half[0] << 32) | half[1];
  }
}

// Warp-wide bound over the sorted prefixes in [lo, n): each round the 32
// lanes probe 32 evenly spaced positions of [lo, hi) (one round trip), a
// ballot keeps the sub-interval that holds the first position whose prefix is
// not below the query's (le = false) or above it (le = true). About log32(n)
// rounds instead of log2(n) dependent steps.
__device__ __forceinline__ int64_t warp_bound(const uint64_t* __restrict__ pre, int64_t n, int K, const uint64_t* qp,
                                              bool le, int64_t lo, int lane) {
  int64_t hi = n;  // answer in [lo, hi]
  while (hi - lo > 0) {
    const int64_t len = hi - lo;
    const int64_t step = (len + 31) / 32;
    const int64_t m = lo + (int64_t)lane * step;
    bool below = false;  // position m lies before the answer
    if (m < hi) {
      const int c = cmp_prefix(pre, n, K, m, qp);
      below = le ? (c <= 0) : (c < 0);
    }
    const uint32_t bm = __ballot_sync(FULL, below);
    const int cnt = __popc(bm);  // lanes 0 .. cnt-1 are below (monotone)
    if (cnt == 0) {
      hi = lo;
    } else {
      const int64_t mlast = lo + (int64_t)(cnt - 1) * step;
      const int64_t nhi = lo + (int64_t)cnt * step;
      lo = mlast + 1;
      hi = nhi < hi ? nhi : hi;
    }
  }
  return lo;
}

// Position of the query in tree t: the lower bound of its full key. qp: K words,
// Yq, Yd: d bytes each, the warp's own.
__device__ __forceinline__ int64_t warp_locate(const SearchArgs& a, int t, const uint8_t* __restrict__ qc,
                                               uint64_t* qp, uint8_t* Yq, uint8_t* Yd, int lane) {
  const int32_t* pi = a.pi + (size_t)t * a.d;
  const uint32_t* rb = a.rbits + (size_t)t * a.W32;
  const uint64_t* pre = a.prefix + (size_t)t * a.K * a.n;
  const uint32_t* sig = a.sigma + (size_t)t * a.n;
  if (a.top) {
    warp_top_prefix(qc, a.bits, a.K, pi, rb, qp, lane);
  } else if (lane == 0) {
    hf_load_coords_codes(qc, a.d, a.bits, a.L, pi, rb, Yq);
    hf_skilling(Yq, a.d, a.L);
    for (int w = 0; w < a.K; ++w) qp[w] = hf_pack_word(Yq, a.d, a.L, w);
  }
  __syncwarp();
  const int64_t lo = warp_bound(pre, a.n, a.K, qp, false, 0, lane);
  int64_t pos = lo;
  // [lo, lo2): positions whose prefix equals the query's
  if (a.K < a.W && lo < a.n && cmp_prefix(pre, a.n, a.K, lo, qp) == 0) {
    const int64_t lo2 = warp_bound(pre, a.n, a.K, qp, true, lo, lane);
    if (lane == 0) {
      // equal prefixes: lower bound by full key inside [lo, lo2)
      hf_load_coords_codes(qc, a.d, a.bits, a.bits, pi, rb, Yq);
      hf_skilling(Yq, a.d, a.bits);
      int64_t l = lo, h = lo2;
      while (l < h) {
        const int64_t mid = (l + h) >> 1;
        hf_load_coords_planes(a.planes, a.n, a.d, a.W32, a.bits, pi, rb, sig[mid], Yd);
        hf_skilling(Yd, a.d, a.bits);
        if (full_key_less(Yd, Yq, a.d, a.bits, a.W)) l = mid + 1;
        else h = mid;
      }
      pos = l;
    }
    pos = __shfl_sync(FULL, pos, 0);
  }
  return pos;
}

// The warp's shared memory (search_per_warp).
struct WarpScratch {
  uint64_t* qp;
  uint32_t* cpid;
  uint8_t *Yq, *Yd;
};
__device__ __forceinline__ WarpScratch warp_scratch(unsigned char* base, int K, int d) {
  WarpScratch w;
  w.qp = reinterpret_cast<uint64_t*>(base);
  w.cpid = reinterpret_cast<uint32_t*>(w.qp + K);
  w.Yq = reinterpret_cast<uint8_t*>(w.cpid + 32);
  w.Yd = w.Yq + d;
  return w;
}

// Positions alone: warp (query, tp) takes trees tp, tp + tsplit, ..., or the one
// tree asked for. Bound by latency (dependent probes of the prefixes, and for
// equal prefixes one lane's keys), so by the warps an SM holds.
__global__ void __launch_bounds__(SWARPS * 32) locate_kernel(SearchArgs a) {
  extern __shared__ __align__(16) unsigned char smraw[];
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const WarpScratch w = warp_scratch(smraw + search_per_warp(a.K, a.d) * wib, a.K, a.d);
  const int64_t wi = (int64_t)blockIdx.x * SWARPS + wib;
  const int64_t qi = wi / a.tsplit;
  if (qi >= a.nq) return;
  const bool one = a.only_tree >= 0;
  const int t_end = one ? a.only_tree + 1 : a.T;
  for (int t = one ? a.only_tree : (int)(wi - qi * a.tsplit); t < t_end; t += a.tsplit) {
    const int64_t pos = warp_locate(a, t, a.qcodes + (size_t)qi * a.d, w.qp, w.Yq, w.Yd, lane);
    if (lane == 0) a.out_pos[one ? (size_t)qi : (size_t)t * a.nq + qi] = pos;
  }
}

// Bitonic sort of one (distance, index) pair per lane across the warp,
// ascending by (distance, index).
__device__ __forceinline__ void warp_sort(float& dv, uint32_t& iv, int lane) {
#pragma unroll
  for (int kk = 2; kk <= 32; kk <<= 1) {
#pragma unroll
    for (int j = kk >> 1; j > 0; j >>= 1) {
      const float od = __shfl_xor_sync(FULL, dv, j);
      const uint32_t oi = __shfl_xor_sync(FULL, iv, j);
      const bool up = (lane & kk) == 0;
      const bool lower = (lane & j) == 0;
      const bool other_less = lessp(od, oi, dv, iv);
      const bool take = (lower == up) ? other_less : !other_less && !(od == dv && oi == iv);
      if (take) {
        dv = od;
        iv = oi;
      }
    }
  }
}

// Transposing butterfly: lane l holds v[u] = its partial for candidate u;
// afterwards v[0] of lane l is the sum over all lanes of the partials for
// candidate l. Step s pairs lanes l and l ^ s; the lane whose bit s is set
// keeps the upper half of the remaining candidates.
__device__ __forceinline__ float warp_transpose_sum(float (&v)[32], int lane) {
#pragma unroll
  for (int s = 16; s >= 1; s >>= 1) {
    const bool up = (lane & s) != 0;
#pragma unroll
    for (int i = 0; i < s; ++i) {
      const float send = up ? v[i] : v[i + s];
      const float keep = up ? v[i + s] : v[i];
      v[i] = keep + __shfl_xor_sync(FULL, send, s);
    }
  }
  return v[0];
}

// Top-k list held across the warp: entry e = 32 s + lane in slot s.
template <int S>
struct WarpList {
  float dv[S];
  uint32_t iv[S];

  __device__ __forceinline__ void init() {
#pragma unroll
    for (int s = 0; s < S; ++s) {
      dv[s] = INFINITY;
      iv[s] = 0xffffffffu;
    }
  }
  // Entry k - 1 (the one a candidate must beat).
  __device__ __forceinline__ void last(int k, float& d, uint32_t& i) const {
    const int s = (k - 1) >> 5, l = (k - 1) & 31;
    float ds = dv[0];
    uint32_t is = iv[0];
#pragma unroll
    for (int t = 1; t < S; ++t)
      if (s == t) {
        ds = dv[t];
        is = iv[t];
      }
    d = __shfl_sync(FULL, ds, l);
    i = __shfl_sync(FULL, is, l);
  }
  __device__ __forceinline__ bool holds(uint32_t ci, int k, int lane) const {
    bool dup = false;
#pragma unroll
    for (int s = 0; s < S; ++s) dup |= 32 * s + lane < k && iv[s] == ci;
    return __any_sync(FULL, dup);
  }
  // Inserts (cd, ci) unless ci is already listed; entries at or beyond k are
  // scratch.
  __device__ __forceinline__ void insert(float cd, uint32_t ci, int k, int lane) {
    bool dup = false;
    int pos = 0;
#pragma unroll
    for (int s = 0; s < S; ++s) {
      const bool valid = 32 * s + lane < k;
      dup |= __ballot_sync(FULL, valid && iv[s] == ci) != 0;
      pos += __popc(__ballot_sync(FULL, valid && lessp(dv[s], iv[s], cd, ci)));
    }
    if (dup) return;
    float cd_prev[S];
    uint32_t ci_prev[S];
#pragma unroll
    for (int s = 0; s < S; ++s) {
      // entry e - 1: lane - 1 of the same slot, or lane 31 of the slot below
      float up_d = __shfl_up_sync(FULL, dv[s], 1);
      uint32_t up_i = __shfl_up_sync(FULL, iv[s], 1);
      const float wrap_d = __shfl_sync(FULL, dv[s > 0 ? s - 1 : 0], 31);
      const uint32_t wrap_i = __shfl_sync(FULL, iv[s > 0 ? s - 1 : 0], 31);
      if (lane == 0) {
        up_d = wrap_d;
        up_i = wrap_i;
      }
      cd_prev[s] = up_d;
      ci_prev[s] = up_i;
    }
#pragma unroll
    for (int s = 0; s < S; ++s) {
      const int e = 32 * s + lane;
      if (e > pos) {
        dv[s] = cd_prev[s];
        iv[s] = ci_prev[s];
      } else if (e == pos) {
        dv[s] = cd;
        iv[s] = ci;
      }
    }
  }
};

__device__ __forceinline__ float bf16_lo(uint32_t u) { return __uint_as_float(u << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t u) { return __uint_as_float(u & 0xffff0000u); }

// acc + (q - (lo, hi))^2 on a pair of floats.
__device__ __forceinline__ uint64_t sq_diff2(uint64_t q, float lo, float hi, uint64_t acc) {
  uint64_t r;
  asm("{\n .reg .b64 v, e;\n mov.b64 v, {%2, %3};\n sub.rn.f32x2 e, %1, v;\n fma.rn.f32x2 %0, e, e, %4;\n}"
      : "=l"(r)
      : "l"(q), "f"(lo), "f"(hi), "l"(acc));
  return r;
}
__device__ __forceinline__ float pair_sum(uint64_t v) {
  return __uint_as_float((uint32_t)v) + __uint_as_float((uint32_t)(v >> 32));
}

// BF16 copy of the points (row pitch dp, a multiple of 64, zero padded) and per
// point an upper bound of |x - copy| (1e-5 above the float32 sum's value; inf
// where a coordinate rounds to inf). One warp per point; d % 4 == 0, rows
// 16-byte aligned.
__global__ void prepare16_kernel(const float* __restrict__ x, int64_t n, int d, int dp, __nv_bfloat16* __restrict__ x16,
                                 float* __restrict__ r16) {
  const int lane = threadIdx.x & 31;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < n; i += nw) {
    float s = 0.f;
    for (int c = 4 * lane; c < dp; c += 128) {
      float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
      if (c < d) v = __ldcs(reinterpret_cast<const float4*>(x + i * d + c));
      const __nv_bfloat162 a = __floats2bfloat162_rn(v.x, v.y), b = __floats2bfloat162_rn(v.z, v.w);
      uint2 o;
      o.x = *reinterpret_cast<const uint32_t*>(&a);
      o.y = *reinterpret_cast<const uint32_t*>(&b);
      *reinterpret_cast<uint2*>(x16 + i * dp + c) = o;
      float e = v.x - bf16_lo(o.x);
      s = fmaf(e, e, s);
      e = v.y - bf16_hi(o.x);
      s = fmaf(e, e, s);
      e = v.z - bf16_lo(o.y);
      s = fmaf(e, e, s);
      e = v.w - bf16_hi(o.y);
      s = fmaf(e, e, s);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(FULL, s, o);
    // squares below the float32 range vanish from the sum: 2^-74 sqrt(d) covers them
    if (lane == 0) r16[i] = sqrtf(s) * 1.00001f + 1e-20f;
  }
}

// Locates and scores: one warp per query, or per part of one.
// Six blocks an SM: 80 registers, 16 rows' loads in flight. Left to itself the
// compiler took the same number and issued the loads one after the other
// (hf_search_static, 10,000 queries, T = 32, w = 8 to 128, d = 64 to 384: a
// geometric mean of 12 % slower at k <= 32, 21 % at k = 64); five blocks (96
// registers) are 9 % faster below 1,000 queries, 7 % slower from 10,000 on.
template <int S>
__global__ void __launch_bounds__(SWARPS * 32, 6) search_kernel(SearchArgs a) {
  extern __shared__ __align__(16) unsigned char smraw[];
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const WarpScratch ws = warp_scratch(smraw + search_per_warp(a.K, a.d) * wib, a.K, a.d);
  uint32_t* cpid = ws.cpid;
  const int parts = a.tsplit * a.csplit;
  const int64_t li = (int64_t)blockIdx.x * SWARPS + wib;  // this warp's list
  const int64_t qi = parts == 1 ? li : li / parts;
  if (qi >= a.nq) return;
  const int part = (int)(li - qi * parts);
  const int tp = part / a.csplit, cp = part - tp * a.csplit;
  const uint8_t* qc = a.qcodes + (size_t)qi * a.d;
  const float* qv = a.q + (size_t)qi * a.d;

  WarpList<S> list;
  list.init();

  for (int t = tp; t < a.T; t += a.tsplit) {
    const uint32_t* sig = a.sigma + (size_t)t * a.n;
    const int64_t pos = warp_locate(a, t, qc, ws.qp, ws.Yq, ws.Yd, lane);
    const int64_t c0 = pos - a.w > 0 ? pos - a.w : 0;
    const int64_t c1 = pos + a.w < a.n ? pos + a.w : a.n;
    for (int64_t cb = c0 + 32 * cp; cb < c1; cb += 32 * a.csplit) {
      const int64_t c = cb + lane;
      uint32_t pid = c < c1 ? __ldg(sig + c) : 0xffffffffu;
      float dist;
      if (a.vec4) {
        cpid[lane] = pid;
        __syncwarp();
        float part[32];
#pragma unroll
        for (int u = 0; u < 32; ++u) part[u] = 0.f;
        for (int m = 4 * lane; m < a.d; m += 128) {
          const float4 qa = __ldg(reinterpret_cast<const float4*>(qv + m));
          // 8 candidate rows per group: all 8 loads are issued before any is
          // used (an empty slot reads the query's own row; its result is
          // discarded)
#pragma unroll
          for (int u0 = 0; u0 < 32; u0 += 16) {
            float4 xb[16];
#pragma unroll
            for (int u = 0; u < 16; ++u) {
              const uint32_t p = cpid[u0 + u];
              const float* row = p != 0xffffffffu ? a.x + (size_t)p * a.d : qv;
              xb[u] = __ldg(reinterpret_cast<const float4*>(row + m));
            }
#pragma unroll
            for (int u = 0; u < 16; ++u) {
              float e = qa.x - xb[u].x;
              float acc = fmaf(e, e, part[u0 + u]);
              e = qa.y - xb[u].y;
              acc = fmaf(e, e, acc);
              e = qa.z - xb[u].z;
              acc = fmaf(e, e, acc);
              e = qa.w - xb[u].w;
              part[u0 + u] = fmaf(e, e, acc);
            }
          }
        }
        dist = warp_transpose_sum(part, lane);
        __syncwarp();
      } else {
        // one lane per candidate over the whole vector
        dist = 0.f;
        if (pid != 0xffffffffu) {
          const float* xv = a.x + (size_t)pid * a.d;
          for (int j = 0; j < a.d; ++j) {
            const float e = __ldg(qv + j) - __ldg(xv + j);
            dist = fmaf(e, e, dist);
          }
        }
      }
      if (pid == 0xffffffffu) dist = INFINITY;
      warp_sort(dist, pid, lane);
      // merge in ascending order; stop at the first that cannot enter
      for (int u = 0; u < 32; ++u) {
        const float cd = __shfl_sync(FULL, dist, u);
        const uint32_t ci = __shfl_sync(FULL, pid, u);
        if (ci == 0xffffffffu) break;
        float kd;
        uint32_t ki;
        list.last(a.k, kd, ki);
        if (!lessp(cd, ci, kd, ki)) break;
        list.insert(cd, ci, a.k, lane);
      }
    }
  }
#pragma unroll
  for (int s = 0; s < S; ++s) {
    const int e = 32 * s + lane;
    if (e < a.k) {
      a.out_idx[(size_t)li * a.k + e] = list.iv[s];
      a.out_dist[(size_t)li * a.k + e] = list.dv[s];
    }
  }
}

// Scores through the half-width screen, the positions known (locate_kernel, in
// a launch of its own: this kernel's registers leave an SM half of the warps
// that hide the locate's latency, which cost batches with few rows per position,
// 64 dimensions or near-duplicates 5 to 20 % of the whole search; 10,000 queries,
// k = 30, both in one kernel and so: 3M x 384, T = 64, w = 50: 12.4, 11.1 ms; 1M
// x 64, T = 64, w = 16: 6.4, 5.1; 300,000 x 384 near-duplicates, T = 64, w = 16:
// 86.4, 57.1).
template <int S>
__global__ void __launch_bounds__(SWARPS * 32) search16_kernel(SearchArgs a) {
  __shared__ uint32_t s_id[SWARPS][32];
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  uint32_t* cpid = s_id[wib];
  const int parts = a.tsplit * a.csplit;
  const int64_t li = (int64_t)blockIdx.x * SWARPS + wib;  // this warp's list
  const int64_t qi = parts == 1 ? li : li / parts;
  if (qi >= a.nq) return;
  const int part = (int)(li - qi * parts);
  const int tp = part / a.csplit, cp = part - tp * a.csplit;
  const float* qv = a.q + (size_t)qi * a.d;

  WarpList<S> list;
  list.init();

  int64_t next = tp < a.T ? __ldg(a.pos + (size_t)tp * a.nq + qi) : 0;
  for (int t = tp; t < a.T; t += a.tsplit) {
    const uint32_t* sig = a.sigma + (size_t)t * a.n;
    const int64_t pos = next;
    if (t + a.tsplit < a.T) next = __ldg(a.pos + (size_t)(t + a.tsplit) * a.nq + qi);
    const int64_t c0 = pos - a.w > 0 ? pos - a.w : 0;
    const int64_t c1 = pos + a.w < a.n ? pos + a.w : a.n;
    for (int64_t cb = c0 + 32 * cp; cb < c1; cb += 32 * a.csplit) {
      const int64_t c = cb + lane;
      const uint32_t pid = c < c1 ? __ldg(sig + c) : 0xffffffffu;
      cpid[lane] = pid;
      const float res = pid != 0xffffffffu ? __ldg(a.r16 + pid) : 0.f;
      __syncwarp();
      const int cnt = (int)(c1 - cb < 32 ? c1 - cb : 32);
      float part[32];
      // 16 rows at a time (none for an empty half): their loads are issued
      // before any is used (an empty slot reads row 0; its result is
      // discarded), two coordinates to an instruction (f32x2), the even and
      // the odd ones' sums apart until the end
#pragma unroll
      for (int u0 = 0; u0 < 32; u0 += 16) {
        uint64_t acc[16];
#pragma unroll
        for (int u = 0; u < 16; ++u) acc[u] = 0;
        if (u0 < cnt) {
          for (int m = 4 * lane; m < a.d; m += 128) {
            const ulonglong2 qa = __ldg(reinterpret_cast<const ulonglong2*>(qv + m));
            uint2 xb[16];
#pragma unroll
            for (int u = 0; u < 16; ++u) {
              const uint32_t p = cpid[u0 + u];
              xb[u] = __ldg(reinterpret_cast<const uint2*>(a.x16 + (size_t)(p != 0xffffffffu ? p : 0u) * a.dp + m));
            }
#pragma unroll
            for (int u = 0; u < 16; ++u) {
              acc[u] = sq_diff2(qa.x, bf16_lo(xb[u].x), bf16_hi(xb[u].x), acc[u]);
              acc[u] = sq_diff2(qa.y, bf16_lo(xb[u].y), bf16_hi(xb[u].y), acc[u]);
            }
          }
        }
#pragma unroll
        for (int u = 0; u < 16; ++u) part[u0 + u] = pair_sum(acc[u]);
      }
      const float near = warp_transpose_sum(part, lane);
      __syncwarp();
      // |q - x| >= |q - copy| - |x - copy|; the sums are within 1e-5 of
      // their values up to d = 4096, also the exact one. A sum that
      // overflowed, or whose squares leave the float32 range, says nothing.
      const float gap = sqrtf(near) * 0.99999f - res;
      const float bound = gap > 1e-12f && near < 1e38f ? gap * gap * 0.99998f : 0.f;
      float kd;
      uint32_t ki;
      list.last(a.k, kd, ki);
      uint32_t todo = __ballot_sync(FULL, pid != 0xffffffffu && !(bound > kd));
      // scores the next NS survivors, their rows' loads in flight together
      auto score = [&](auto count) {
        constexpr int NS = decltype(count)::value;
        uint32_t ci[NS];
        float cd[NS];
#pragma unroll
        for (int u = 0; u < NS; ++u) {
          const int src = todo ? __ffs(todo) - 1 : 0;
          const bool some = todo != 0;
          todo &= todo - 1;
          const uint32_t id = __shfl_sync(FULL, pid, src);
          const bool out = __shfl_sync(FULL, bound, src) > kd;
          ci[u] = some && !out && !list.holds(id, a.k, lane) ? id : 0xffffffffu;
          cd[u] = 0.f;
        }
        for (int m = 4 * lane; m < a.d; m += 128) {
          const float4 qa = __ldg(reinterpret_cast<const float4*>(qv + m));
          float4 xv[NS];
#pragma unroll
          for (int u = 0; u < NS; ++u)
            xv[u] = ci[u] != 0xffffffffu ? __ldg(reinterpret_cast<const float4*>(a.x + (size_t)ci[u] * a.d + m)) : qa;
#pragma unroll
          for (int u = 0; u < NS; ++u) {
            float e = qa.x - xv[u].x;
            cd[u] = fmaf(e, e, cd[u]);
            e = qa.y - xv[u].y;
            cd[u] = fmaf(e, e, cd[u]);
            e = qa.z - xv[u].z;
            cd[u] = fmaf(e, e, cd[u]);
            e = qa.w - xv[u].w;
            cd[u] = fmaf(e, e, cd[u]);
          }
        }
        // the lanes' partials in warp_transpose_sum's tree
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
          for (int u = 0; u < NS; ++u) cd[u] += __shfl_xor_sync(FULL, cd[u], o);
#pragma unroll
        for (int u = 0; u < NS; ++u)
          if (ci[u] != 0xffffffffu && lessp(cd[u], ci[u], kd, ki)) {
            list.insert(cd[u], ci[u], a.k, lane);
            list.last(a.k, kd, ki);
          }
      };
      // one at a time once they are few: the list's last distance, which each may
      // lower, spares the next one its row
      while (todo) {
        if (__popc(todo) >= 3) score(std::integral_constant<int, 4>{});
        else score(std::integral_constant<int, 1>{});
      }
    }
  }
#pragma unroll
  for (int s = 0; s < S; ++s) {
    const int e = 32 * s + lane;
    if (e < a.k) {
      a.out_idx[(size_t)li * a.k + e] = list.iv[s];
      a.out_dist[(size_t)li * a.k + e] = list.dv[s];
    }
  }
}

// Top k of a query's part lists (each ascending): one warp per query, the
// parts in turn, 32 entries at a time until the first that cannot enter. A
// point found by several parts has the same distance in each; the insertion
// drops the repeats.
template <int S>
__global__ void __launch_bounds__(SWARPS * 32)
merge_parts_kernel(const uint32_t* __restrict__ pidx, const float* __restrict__ pdist, int64_t nq, int parts, int k,
                   uint32_t* __restrict__ out_idx, float* __restrict__ out_dist) {
  const int lane = threadIdx.x & 31;
  const int64_t qi = (int64_t)blockIdx.x * SWARPS + (threadIdx.x >> 5);
  if (qi >= nq) return;
  WarpList<S> list;
  list.init();
  const int64_t total = (int64_t)parts * k;
  const uint32_t* qidx = pidx + (size_t)qi * total;
  const float* qdist = pdist + (size_t)qi * total;
  uint32_t nid = lane < k ? __ldg(qidx + lane) : 0xffffffffu;  // the next part's first entries are in flight
  float nd = lane < k ? __ldg(qdist + lane) : INFINITY;
  for (int p = 0; p < parts; ++p) {
    bool more = true;
    for (int e0 = 0; e0 < k && more; e0 += 32) {
      uint32_t id = nid;
      float dv = nd;
      if (e0) {
        id = e0 + lane < k ? __ldg(qidx + (size_t)p * k + e0 + lane) : 0xffffffffu;
        dv = e0 + lane < k ? __ldg(qdist + (size_t)p * k + e0 + lane) : INFINITY;
      } else if (p + 1 < parts) {
        nid = lane < k ? __ldg(qidx + (size_t)(p + 1) * k + lane) : 0xffffffffu;
        nd = lane < k ? __ldg(qdist + (size_t)(p + 1) * k + lane) : INFINITY;
      }
      for (int u = 0; u < 32; ++u) {
        const float cd = __shfl_sync(FULL, dv, u);
        const uint32_t ci = __shfl_sync(FULL, id, u);
        float kd;
        uint32_t ki;
        list.last(k, kd, ki);
        if (ci == 0xffffffffu || !lessp(cd, ci, kd, ki)) {
          more = false;
          break;
        }
        list.insert(cd, ci, k, lane);
      }
    }
  }
#pragma unroll
  for (int s = 0; s < S; ++s) {
    const int e = 32 * s + lane;
    if (e < k) {
      out_idx[(size_t)qi * k + e] = list.iv[s];
      out_dist[(size_t)qi * k + e] = list.dv[s];
    }
  }
}

template <int S>
int launch_s(const SearchArgs& a, size_t smem, cudaStream_t s) {
  const unsigned blocks = hf_blocks(a.nq * a.tsplit * a.csplit, SWARPS);
  if (a.pos) {
    search16_kernel<S><<<blocks, SWARPS * 32, 0, s>>>(a);
    hf_after_launch("search16_kernel", s);
    return HF_OK;
  }
  if (smem > 48 * 1024 && cudaFuncSetAttribute((const void*)search_kernel<S>,
                                               cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
    return HF_ECUDA;
  search_kernel<S><<<blocks, SWARPS * 32, smem, s>>>(a);
  hf_after_launch("search_kernel", s);
  return HF_OK;
}

int launch_locate(const SearchArgs& a, size_t smem, cudaStream_t s) {
  if (smem > 48 * 1024 && cudaFuncSetAttribute((const void*)locate_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               (int)smem) != cudaSuccess)
    return HF_ECUDA;
  locate_kernel<<<hf_blocks(a.nq * a.tsplit, SWARPS), SWARPS * 32, smem, s>>>(a);
  hf_after_launch("locate_kernel", s);
  return HF_OK;
}

template <int S>
void launch_merge(const SearchArgs& a, uint32_t* out_idx, float* out_dist, cudaStream_t s) {
  merge_parts_kernel<S><<<hf_blocks(a.nq, SWARPS), SWARPS * 32, 0, s>>>(a.out_idx, a.out_dist, a.nq,
                                                                       a.tsplit * a.csplit, a.k, out_idx, out_dist);
  hf_after_launch("merge_parts_kernel", s);
}

// Parts per query. One warp walks all T trees of a query in T dependent steps
// (key, probes, rows), which is the whole time of a small batch (5 queries, T =
// 32, w = 32, 200,000 x 384: 1001 us a call, 107 split into 64 parts each). The
// trees, then the chunks of a window, go to as many warps as give the chip
// SPLIT_WARPS of them; from half that many queries on the batch fills the chip
// by itself. search_parts sizes the part lists from the same split.
constexpr int64_t SPLIT_WARPS = 152 * 16;

void search_split(int64_t nq, int T, int w, int* tsplit, int* csplit) {
  const int64_t want = SPLIT_WARPS / nq;
  *tsplit = *csplit = 1;
  if (want < 2) return;
  *tsplit = (int)(want < T ? want : T);
  const int64_t chunks = ((int64_t)2 * w + 31) / 32, rest = want / *tsplit;
  *csplit = (int)(rest < chunks ? rest : chunks);
  if (*csplit > 4) *csplit = 4;  // the merge walks the parts one by one
}

}  // namespace

void launch_prepare16(const float* x, int64_t n, int d, void* x16, float* r16, cudaStream_t s) {
  prepare16_kernel<<<hf_blocks(n * 32, 256, 152 * 16), 256, 0, s>>>(x, n, d, (d + 63) / 64 * 64,
                                                                   static_cast<__nv_bfloat16*>(x16), r16);
  hf_after_launch("prepare16_kernel", s);
}

int64_t search_parts(const hf_forest* f, int64_t nq, int w) {
  int ts, cs;
  search_split(nq, f->T, w, &ts, &cs);
  return (int64_t)ts * cs;
}

namespace {

SearchArgs search_args(const hf_forest* f, const float* q, const uint8_t* qcodes, int64_t nq, int k, int w) {
  SearchArgs a{};
  a.x = f->x;
  a.n = f->n;
  a.d = f->d;
  a.bits = f->bits;
  a.K = f->K;
  a.L = f->L;
  a.W = f->W;
  a.W32 = f->W32;
  a.T = f->T;
  a.planes = f->planes;
  a.pi = f->pi;
  a.rbits = f->rbits;
  a.prefix = f->prefix;
  a.sigma = f->sigma;
  a.q = q;
  a.qcodes = qcodes;
  a.nq = nq;
  a.k = k;
  a.w = w;
  a.only_tree = -1;
  a.vec4 = (f->d % 4 == 0) && ((reinterpret_cast<uintptr_t>(f->x) & 15) == 0) &&
           ((reinterpret_cast<uintptr_t>(q) & 15) == 0);
  a.top = f->d >= 64 * f->K;
  a.dp = (f->d + 63) / 64 * 64;
  a.tsplit = a.csplit = 1;
  return a;
}

}  // namespace

int launch_positions(const hf_forest* f, const float* q, const uint8_t* qcodes, int64_t nq, int tree, int64_t* out_pos,
                     cudaStream_t s) {
  SearchArgs a = search_args(f, q, qcodes, nq, 1, 1);
  a.out_pos = out_pos;
  a.only_tree = tree;
  if (tree < 0) {
    // trees are independent, nothing to merge
    int cs;
    search_split(nq, f->T, 1, &a.tsplit, &cs);
  }
  const int rc = launch_locate(a, search_per_warp(f->K, f->d) * SWARPS, s);
  if (rc != HF_OK) return rc;
  return cudaGetLastError() == cudaSuccess ? HF_OK : HF_ECUDA;
}

int64_t search16_slice(int64_t nq, int T) {
  int64_t slice = ((int64_t)64 << 20) / (8 * (int64_t)T);
  if (slice < 2048) slice = 2048;
  return slice < nq ? slice : nq;
}

int launch_search(const hf_forest* f, const float* q, const uint8_t* qcodes, int64_t nq, int k, int w,
                  uint32_t* out_idx, float* out_dist, cudaStream_t s, uint32_t* part_idx, float* part_dist,
                  int64_t* pos16) {
  if (k < 1 || k > 64) return HF_EINVAL;
  const size_t smem = search_per_warp(f->K, f->d) * SWARPS;
  const int64_t slice = pos16 ? search16_slice(nq, f->T) : nq;
  for (int64_t q0 = 0; q0 < nq; q0 += slice) {
    const int64_t m = nq - q0 < slice ? nq - q0 : slice;
    SearchArgs a = search_args(f, q + (size_t)q0 * f->d, qcodes + (size_t)q0 * f->d, m, k, w);
    uint32_t* oi = a.out_idx = out_idx + (size_t)q0 * k;
    float* od = a.out_dist = out_dist + (size_t)q0 * k;
    int rc = HF_OK;
    if (pos16 && a.vec4 && f->x16) {
      a.out_pos = pos16;
      a.tsplit = f->T;
      rc = launch_locate(a, smem, s);
      a.tsplit = 1;
      a.pos = pos16;
      a.x16 = static_cast<const __nv_bfloat16*>(f->x16);
      a.r16 = f->r16;
    }
    if (part_idx) search_split(m, f->T, w, &a.tsplit, &a.csplit);
    const bool parts = a.tsplit * a.csplit > 1;
    if (parts) {
      a.out_idx = part_idx;
      a.out_dist = part_dist;
    }
    if (rc == HF_OK) rc = k <= 32 ? launch_s<1>(a, smem, s) : launch_s<2>(a, smem, s);
    if (rc != HF_OK) return rc;
    if (parts) {
      if (k <= 32) launch_merge<1>(a, oi, od, s);
      else launch_merge<2>(a, oi, od, s);
    }
  }
  return cudaGetLastError() == cudaSuccess ? HF_OK : HF_ECUDA;
}

// ---------------------------------------------------------------------------
// Search with the second-stage filter and the master-order expansion
// (Algorithm 1, both filters).
//
// One warp per query, after the positions of every tree are known:
//  * Hamming stage: the window candidates of each tree go 32 at a time, one
//    per lane; a lane XORs its candidate's sketch with the query's (held in
//    shared memory) and counts the bits; the 32 counts are sorted across the
//    warp and merged into a warp-held list of the k2 smallest (Hamming
//    distance, index), duplicates across trees dropped on insertion.
//  * Expansion: entry e of the expanded set is survivor e / (2h + 1) shifted by
//    e % (2h + 1) - h positions in the master order (order 0), clipped. The
//    rows come from the master-ordered copy of the points, so the 2h + 1 rows
//    of one survivor are adjacent in memory.
//  * Final stage: the expanded entries are scored with the same float32
//    exact-difference distance and transposing butterfly as the plain search
//    and merged into the warp-held top-k list.
// ---------------------------------------------------------------------------
namespace {

constexpr int SK_MAX_WORDS = 16;  // sketches up to 1024 bits

struct SketchSearchArgs {
  const float* q;
  int64_t nq;
  int d;
  const float* xm;         // n x d, row p = point sig0[p]
  const uint32_t* sig0;    // master order
  const uint32_t* posm;    // inverse of the master order
  const uint32_t* sigma;   // T x n orders
  const int64_t* pos;      // T x nq lower-bound positions
  const uint64_t* sk;      // n x words
  const uint64_t* qsk;     // nq x words
  int words;
  int64_t n;
  int T, w, k2, h, k;
  uint32_t* out_idx;
  float* out_dist;
  int vec4;
};

template <int S2, int S>
__global__ void __launch_bounds__(SWARPS * 32) sketch_search_kernel(SketchSearchArgs a) {
  __shared__ uint64_t s_q[SWARPS][SK_MAX_WORDS];
  __shared__ uint32_t s_c2[SWARPS][32 * S2];
  __shared__ uint32_t s_id[SWARPS][32];
  __shared__ uint32_t s_row[SWARPS][32];
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const int64_t qi = (int64_t)blockIdx.x * SWARPS + wib;
  if (qi >= a.nq) return;
  if (lane < a.words) s_q[wib][lane] = a.qsk[(size_t)qi * a.words + lane];
  __syncwarp();

  // Hamming stage
  WarpList<S2> l2;
  l2.init();
  for (int t = 0; t < a.T; ++t) {
    const int64_t pos = a.pos[(size_t)t * a.nq + qi];
    const uint32_t* sig = a.sigma + (size_t)t * a.n;
    const int64_t c0 = pos - a.w > 0 ? pos - a.w : 0;
    const int64_t c1 = pos + a.w < a.n ? pos + a.w : a.n;
    for (int64_t cb = c0; cb < c1; cb += 32) {
      const int64_t c = cb + lane;
      uint32_t pid = c < c1 ? __ldg(sig + c) : 0xffffffffu;
      float hd = INFINITY;
      if (pid != 0xffffffffu) {
        const uint64_t* row = a.sk + (size_t)pid * a.words;
        int hm = 0;
        for (int u = 0; u < a.words; ++u) hm += __popcll(s_q[wib][u] ^ __ldg(row + u));
        hd = (float)hm;
      }
      warp_sort(hd, pid, lane);
      for (int u = 0; u < 32; ++u) {
        const float cd = __shfl_sync(FULL, hd, u);
        const uint32_t ci = __shfl_sync(FULL, pid, u);
        if (ci == 0xffffffffu) break;
        float kd;
        uint32_t ki;
        l2.last(a.k2, kd, ki);
        if (!lessp(cd, ci, kd, ki)) break;
        l2.insert(cd, ci, a.k2, lane);
      }
    }
  }
#pragma unroll
  for (int s2 = 0; s2 < S2; ++s2) s_c2[wib][32 * s2 + lane] = 32 * s2 + lane < a.k2 ? l2.iv[s2] : 0xffffffffu;
  __syncwarp();

  // expansion and final stage
  const float* qv = a.q + (size_t)qi * a.d;
  WarpList<S> list;
  list.init();
  const int span = 2 * a.h + 1;
  const int64_t E = (int64_t)a.k2 * span;
  for (int64_t eb = 0; eb < E; eb += 32) {
    const int64_t e = eb + lane;
    uint32_t pid = 0xffffffffu, row = 0;
    if (e < E) {
      const int u = (int)(e / span), o = (int)(e % span) - a.h;
      const uint32_t c = s_c2[wib][u];
      if (c != 0xffffffffu) {
        const int64_t p = (int64_t)__ldg(a.posm + c) + o;
        if (p >= 0 && p < a.n) {
          row = (uint32_t)p;
          pid = __ldg(a.sig0 + p);
        }
      }
    }
    float dist;
    if (a.vec4) {
      s_id[wib][lane] = pid;
      s_row[wib][lane] = row;
      __syncwarp();
      float part[32];
#pragma unroll
      for (int u = 0; u < 32; ++u) part[u] = 0.f;
      for (int m = 4 * lane; m < a.d; m += 128) {
        const float4 qa = __ldg(reinterpret_cast<const float4*>(qv + m));
#pragma unroll
        for (int u0 = 0; u0 < 32; u0 += 16) {
          float4 xb[16];
#pragma unroll
          for (int u = 0; u < 16; ++u) {
            // an empty entry reads master row 0; its result is discarded
            xb[u] = __ldg(reinterpret_cast<const float4*>(a.xm + (size_t)s_row[wib][u0 + u] * a.d + m));
          }
#pragma unroll
          for (int u = 0; u < 16; ++u) {
            float ee = qa.x - xb[u].x;
            float acc = fmaf(ee, ee, part[u0 + u]);
            ee = qa.y - xb[u].y;
            acc = fmaf(ee, ee, acc);
            ee = qa.z - xb[u].z;
            acc = fmaf(ee, ee, acc);
            ee = qa.w - xb[u].w;
            part[u0 + u] = fmaf(ee, ee, acc);
          }
        }
      }
      dist = warp_transpose_sum(part, lane);
      __syncwarp();
    } else {
      dist = 0.f;
      if (pid != 0xffffffffu) {
        const float* xv = a.xm + (size_t)row * a.d;
        for (int j = 0; j < a.d; ++j) {
          const float ee = __ldg(qv + j) - __ldg(xv + j);
          dist = fmaf(ee, ee, dist);
        }
      }
    }
    if (pid == 0xffffffffu) dist = INFINITY;
    warp_sort(dist, pid, lane);
    for (int u = 0; u < 32; ++u) {
      const float cd = __shfl_sync(FULL, dist, u);
      const uint32_t ci = __shfl_sync(FULL, pid, u);
      if (ci == 0xffffffffu) break;
      float kd;
      uint32_t ki;
      list.last(a.k, kd, ki);
      if (!lessp(cd, ci, kd, ki)) break;
      list.insert(cd, ci, a.k, lane);
    }
  }
#pragma unroll
  for (int s2 = 0; s2 < S; ++s2) {
    const int e = 32 * s2 + lane;
    if (e < a.k) {
      a.out_idx[(size_t)qi * a.k + e] = list.iv[s2];
      a.out_dist[(size_t)qi * a.k + e] = list.dv[s2];
    }
  }
}

// Master-ordered copy of the points and the inverse of the master order.
__global__ void master_layout_kernel(const float* __restrict__ x, int64_t n, int d, const uint32_t* __restrict__ sig0,
                                     float* __restrict__ xm, uint32_t* __restrict__ posm) {
  const int64_t total = n * d;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t p = e / d;
    const int j = (int)(e - p * d);
    const uint32_t id = __ldg(sig0 + p);
    xm[e] = __ldg(x + (size_t)id * d + j);
    if (j == 0) posm[id] = (uint32_t)p;
  }
}

// Exact k nearest neighbours of given rows among the points of their own set
// (the whole matrix when unsegmented), the row itself excluded: one warp per
// row, every point of the set scored 32 at a time with the search's float32
// exact-difference distance and merged into the warp-held list.
template <int S>
__global__ void __launch_bounds__(SWARPS * 32)
exact_rows_kernel(const float* __restrict__ x, int64_t n, int d, const int64_t* __restrict__ rows, int nrows,
                  const uint32_t* __restrict__ segr, const int64_t* __restrict__ segoff, int k, int vec4,
                  uint32_t* __restrict__ out_idx, float* __restrict__ out_dist) {
  __shared__ uint32_t s_id[SWARPS][32];
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const int64_t wi = (int64_t)blockIdx.x * SWARPS + wib;
  if (wi >= nrows) return;
  const int64_t r = rows[wi];
  const float* qv = x + (size_t)r * d;
  int64_t lo = 0, hi = n;
  if (segr) {
    const uint32_t sg = __ldg(segr + r);
    lo = __ldg(segoff + sg);
    hi = __ldg(segoff + sg + 1);
  }
  WarpList<S> list;
  list.init();
  for (int64_t cb = lo; cb < hi; cb += 32) {
    const int64_t c = cb + lane;
    uint32_t pid = (c < hi && c != r) ? (uint32_t)c : 0xffffffffu;
    float dist;
    if (vec4) {
      s_id[wib][lane] = pid;
      __syncwarp();
      float part[32];
#pragma unroll
      for (int u = 0; u < 32; ++u) part[u] = 0.f;
      for (int m = 4 * lane; m < d; m += 128) {
        const float4 qa = __ldg(reinterpret_cast<const float4*>(qv + m));
#pragma unroll
        for (int u0 = 0; u0 < 32; u0 += 16) {
          float4 xb[16];
#pragma unroll
          for (int u = 0; u < 16; ++u) {
            const uint32_t p = s_id[wib][u0 + u];
            const float* row = p != 0xffffffffu ? x + (size_t)p * d : qv;
            xb[u] = __ldg(reinterpret_cast<const float4*>(row + m));
          }
#pragma unroll
          for (int u = 0; u < 16; ++u) {
            float e = qa.x - xb[u].x;
            float acc = fmaf(e, e, part[u0 + u]);
            e = qa.y - xb[u].y;
            acc = fmaf(e, e, acc);
            e = qa.z - xb[u].z;
            acc = fmaf(e, e, acc);
            e = qa.w - xb[u].w;
            part[u0 + u] = fmaf(e, e, acc);
          }
        }
      }
      dist = warp_transpose_sum(part, lane);
      __syncwarp();
    } else {
      dist = 0.f;
      if (pid != 0xffffffffu) {
        const float* xv = x + (size_t)pid * d;
        for (int j = 0; j < d; ++j) {
          const float e = __ldg(qv + j) - __ldg(xv + j);
          dist = fmaf(e, e, dist);
        }
      }
    }
    if (pid == 0xffffffffu) dist = INFINITY;
    warp_sort(dist, pid, lane);
    for (int u = 0; u < 32; ++u) {
      const float cd = __shfl_sync(FULL, dist, u);
      const uint32_t ci = __shfl_sync(FULL, pid, u);
      if (ci == 0xffffffffu) break;
      float kd;
      uint32_t ki;
      list.last(k, kd, ki);
      if (!lessp(cd, ci, kd, ki)) break;
      list.insert(cd, ci, k, lane);
    }
  }
#pragma unroll
  for (int s2 = 0; s2 < S; ++s2) {
    const int e = 32 * s2 + lane;
    if (e < k) {
      out_idx[(size_t)wi * k + e] = list.iv[s2];
      out_dist[(size_t)wi * k + e] = list.dv[s2];
    }
  }
}

// out[j][c] = lists[rows[j]][c] for c < k (lists have kp slots per row).
__global__ void gather_list_rows_kernel(const uint32_t* __restrict__ lists, int kp, const int64_t* __restrict__ rows,
                                        int nrows, int k, uint32_t* __restrict__ out) {
  const int64_t total = (int64_t)nrows * k;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t j = e / k;
    out[e] = lists[(size_t)rows[j] * kp + (e - j * k)];
  }
}

template <int S2, int S>
int launch_ss(const SketchSearchArgs& a, cudaStream_t s) {
  sketch_search_kernel<S2, S><<<hf_blocks(a.nq, SWARPS), SWARPS * 32, 0, s>>>(a);
  hf_after_launch("sketch_search_kernel", s);
  return HF_OK;
}

template <int S>
int launch_ss_k2(const SketchSearchArgs& a, cudaStream_t s) {
  if (a.k2 <= 32) return launch_ss<1, S>(a, s);
  if (a.k2 <= 64) return launch_ss<2, S>(a, s);
  if (a.k2 <= 128) return launch_ss<4, S>(a, s);
  if (a.k2 <= 256) return launch_ss<8, S>(a, s);
  if (a.k2 <= 512) return launch_ss<16, S>(a, s);
  return launch_ss<32, S>(a, s);
}

}  // namespace

int launch_exact_rows(const hf_forest* f, const int64_t* rows, int nrows, int k, uint32_t* out_idx, float* out_dist,
                      cudaStream_t s) {
  if (k < 1 || k > 64 || nrows < 1) return HF_EINVAL;
  const int vec4 = f->d % 4 == 0 && (reinterpret_cast<uintptr_t>(f->x) & 15) == 0;
  const uint32_t* segr = f->nseg > 1 ? f->seg : nullptr;
  const int64_t* segoff = f->nseg > 1 ? f->seg_off : nullptr;
  if (k <= 32)
    exact_rows_kernel<1><<<hf_blocks(nrows, SWARPS), SWARPS * 32, 0, s>>>(f->x, f->n, f->d, rows, nrows, segr, segoff,
                                                                          k, vec4, out_idx, out_dist);
  else
    exact_rows_kernel<2><<<hf_blocks(nrows, SWARPS), SWARPS * 32, 0, s>>>(f->x, f->n, f->d, rows, nrows, segr, segoff,
                                                                          k, vec4, out_idx, out_dist);
  hf_after_launch("exact_rows_kernel", s);
  return HF_OK;
}

void launch_gather_list_rows(const uint32_t* lists, int kp, const int64_t* rows, int nrows, int k, uint32_t* out,
                             cudaStream_t s) {
  gather_list_rows_kernel<<<hf_blocks((int64_t)nrows * k, 256, 152 * 4), 256, 0, s>>>(lists, kp, rows, nrows, k, out);
  hf_after_launch("gather_list_rows_kernel", s);
}

void launch_master_layout(const float* x, int64_t n, int d, const uint32_t* sig0, float* xm, uint32_t* posm,
                          cudaStream_t s) {
  master_layout_kernel<<<hf_blocks(n * d, 256, 152 * 16), 256, 0, s>>>(x, n, d, sig0, xm, posm);
  hf_after_launch("master_layout_kernel", s);
}

int launch_sketch_search(const hf_forest* f, const float* q, int64_t nq, const int64_t* pos, const uint64_t* qsk,
                         int k, int w, int k2, int h, uint32_t* out_idx, float* out_dist, cudaStream_t s) {
  if (k < 1 || k > 64 || k2 < 1 || k2 > HF_MAX_K2 || h < 0 || !f->sketch || !f->xm || !f->posm) return HF_EINVAL;
  const int words = f->sketch_bits / 64;
  if (words < 1 || words > SK_MAX_WORDS) return HF_EINVAL;
  SketchSearchArgs a;
  a.q = q;
  a.nq = nq;
  a.d = f->d;
  a.xm = f->xm;
  a.sig0 = f->sigma;
  a.posm = f->posm;
  a.sigma = f->sigma;
  a.pos = pos;
  a.sk = f->sketch;
  a.qsk = qsk;
  a.words = words;
  a.n = f->n;
  a.T = f->T;
  a.w = w;
  a.k2 = k2;
  a.h = h;
  a.k = k;
  a.out_idx = out_idx;
  a.out_dist = out_dist;
  a.vec4 = (f->d % 4 == 0) && ((reinterpret_cast<uintptr_t>(f->xm) & 15) == 0) &&
           ((reinterpret_cast<uintptr_t>(q) & 15) == 0);
  return k <= 32 ? launch_ss_k2<1>(a, s) : launch_ss_k2<2>(a, s);
}

// ---------------------------------------------------------------------------
// Allocation-free search.
//
// hf_search allocates a device buffer for the queries' quantized codes on
// every call. Some callers cannot allocate device memory while they run: a
// serving process that holds a fixed memory budget carved out up front, a
// host runtime that owns all device memory through its own pool, or a worker
// that must not take the allocator's locks on its latency path. For them,
// hf_search_static keeps that scratch in a fixed array that lives in this
// library's device image: every GPU that loads the library holds
// HF_STATIC_QUERY_BYTES of it until the process exits.
//
// The array's host-side name is only a stand-in for the device symbol, so the
// host looks up its device address with cudaGetSymbolAddress, once per
// device, with that device current, and passes that address to the kernels.
// ---------------------------------------------------------------------------
#include <mutex>

namespace {

__device__ __align__(256) uint8_t g_static_qcodes[HF_STATIC_QUERY_BYTES];

constexpr int kMaxDevices = 64;
std::mutex g_static_mu;
uint8_t* g_static_addr[kMaxDevices] = {};

// Device address of g_static_qcodes on the current device (looked up on the
// first call per device).
int static_qcodes_address(uint8_t** out) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) {
    cudaGetLastError();
    return HF_ECUDA;
  }
  std::lock_guard<std::mutex> lock(g_static_mu);
  if (!g_static_addr[dev]) {
    void* p = nullptr;
    if (cudaGetSymbolAddress(&p, g_static_qcodes) != cudaSuccess || !p) {
      cudaGetLastError();
      return HF_ECUDA;
    }
    g_static_addr[dev] = static_cast<uint8_t*>(p);
  }
  *out = g_static_addr[dev];
  return HF_OK;
}

bool on_device(const void* p) {
  cudaPointerAttributes at;
  if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return at.type == cudaMemoryTypeDevice || at.type == cudaMemoryTypeManaged;
}

}  // namespace

extern "C" int hf_search_static(hf_forest* f, const float* queries, int64_t nq, int32_t k, int32_t w,
                                int32_t* out_idx, float* out_dist, void* stream) {
  if (!f || nq < 0 || k < 1 || k > HF_MAX_K || w < 1) return HF_EINVAL;
  if (f->mode == 3) return HF_ENOTIMPL;  // the sketch form needs per-call scratch
  if (f->nseg > 1) return HF_ENOTIMPL;   // segmented orders carry no search prefixes
  if (nq == 0) return HF_OK;
  if (!queries || !out_idx || !out_dist) return HF_EINVAL;
  if ((uint64_t)nq * (uint64_t)f->d > (uint64_t)HF_STATIC_QUERY_BYTES) return HF_EINVAL;
  if (!on_device(queries) || !on_device(out_idx) || !on_device(out_dist)) return HF_EINVAL;
  uint8_t* qc = nullptr;
  int rc = static_qcodes_address(&qc);
  if (rc != HF_OK) return rc;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  cudaGetLastError();  // an earlier call's error was reported by that call
  launch_quantize_codes(queries, nq, f->d, f->lo, f->scale, f->bits, qc, f->err, s);
  rc = launch_search(f, queries, qc, nq, k, w, reinterpret_cast<uint32_t*>(out_idx), out_dist, s);
  // the same synchronisation and status mapping as every other entry point
  const int rc2 = hf_finish(f, s);
  return rc != HF_OK ? rc : rc2;
}
