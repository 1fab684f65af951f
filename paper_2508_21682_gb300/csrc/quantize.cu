// Per-axis range and b-bit quantization of the points.
//
// The paper quantizes vectors for its distance stage (Section 3, 4-bit codes)
// but does not say how coordinates are discretised for the Hilbert sort. This
// library fixes: lo_j = min_i x_ij, hi_j = max_i x_ij, scale_j =
// (float)(2^b / (double)(float)(hi_j - lo_j)) (0 for a flat axis), and
// code = clamp(floor(fl32(fl32(x - lo) * scale)), 0, 2^b - 1), each step a
// separately rounded float32 operation (__fsub_rn / __fmul_rn, never fused).
//
// Codes are stored as b bit planes, plane 0 holding the most significant bit:
// planes[l][i][m] bit j = bit (b-1-l) of the code of coordinate 32m + j of
// point i. A key prefix that needs only the top level reads one plane
// (d/8 bytes per point) instead of the whole code row.
#include <cuda_runtime.h>
#include <math.h>

#include "hf_internal.cuh"

namespace {

constexpr int RANGE_THREADS = 256;

// Each thread owns one column group of `vec` consecutive columns for the whole
// run, because the total thread count is a multiple of d / vec; it keeps a
// running min / max and writes them to partial[thread].
template <int VEC>
__global__ void range_partial_kernel(const float* __restrict__ x, int64_t total_vec, int d,
                                     int64_t nthreads, float* __restrict__ pmin,
                                     float* __restrict__ pmax, int* __restrict__ err) {
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= nthreads) return;
  float mn[VEC], mx[VEC];
#pragma unroll
  for (int v = 0; v < VEC; ++v) {
    mn[v] = INFINITY;
    mx[v] = -INFINITY;
  }
  bool bad = false;
  for (int64_t e = t; e < total_vec; e += nthreads) {
    if (VEC == 4) {
      const float4 q = __ldg(reinterpret_cast<const float4*>(x) + e);
      const float vals[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
      for (int v = 0; v < VEC; ++v) {
        bad |= !isfinite(vals[v]);
        mn[v] = fminf(mn[v], vals[v]);
        mx[v] = fmaxf(mx[v], vals[v]);
      }
    } else {
      const float val = __ldg(x + e);
      bad |= !isfinite(val);
      mn[0] = fminf(mn[0], val);
      mx[0] = fmaxf(mx[0], val);
    }
  }
  if (bad) hf_raise(err, HF_ERRBIT_NONFINITE);
#pragma unroll
  for (int v = 0; v < VEC; ++v) {
    pmin[t * VEC + v] = mn[v];
    pmax[t * VEC + v] = mx[v];
  }
}

// One block per column c: the partials of threads t with (t*VEC) % d == c - v
// are reduced by the block's threads, then across the block.
__global__ void range_final_kernel(const float* __restrict__ pmin, const float* __restrict__ pmax,
                                   int64_t nthreads, int vec, int d, int bits,
                                   float* __restrict__ lo, float* __restrict__ scale) {
  __shared__ float smn[32], smx[32];
  const int c = blockIdx.x;
  const int groups = d / vec;  // threads per "row" of column groups
  const int g = c / vec, v = c % vec;
  float mn = INFINITY, mx = -INFINITY;
  for (int64_t t = g + (int64_t)threadIdx.x * groups; t < nthreads; t += (int64_t)blockDim.x * groups) {
    mn = fminf(mn, pmin[t * vec + v]);
    mx = fmaxf(mx, pmax[t * vec + v]);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    mn = fminf(mn, __shfl_xor_sync(0xffffffffu, mn, o));
    mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  }
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (lane == 0) {
    smn[wid] = mn;
    smx[wid] = mx;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w) {
      mn = fminf(mn, smn[w]);
      mx = fmaxf(mx, smx[w]);
    }
    lo[c] = mn;
    const float width = __fsub_rn(mx, mn);
    scale[c] = width > 0.0f ? (float)((double)(1u << bits) / (double)width) : 0.0f;
  }
}

__device__ __forceinline__ uint32_t quantize_one(float x, float lo, float scale, int bits) {
  const float diff = __fsub_rn(x, lo);
  const float prod = __fmul_rn(diff, scale);
  const float fl = floorf(prod);
  const float top = (float)((1u << bits) - 1u);
  const float cl = fminf(fmaxf(fl, 0.0f), top);
  return (uint32_t)cl;
}

// 8 x 8 bit-matrix transpose of a 64-bit word: bit c of byte u moves to
// bit u of byte c (delta swaps of 7, 14 and 28 positions).
__device__ __forceinline__ uint64_t transpose8x8(uint64_t x) {
  uint64_t t = (x ^ (x >> 7)) & 0x00AA00AA00AA00AAull;
  x = x ^ t ^ (t << 7);
  t = (x ^ (x >> 14)) & 0x0000CCCC0000CCCCull;
  x = x ^ t ^ (t << 14);
  t = (x ^ (x >> 28)) & 0x00000000F0F0F0F0ull;
  x = x ^ t ^ (t << 28);
  return x;
}

// A warp takes pb consecutive points at a time. Lane by lane it goes through
// their groups of 8 consecutive coordinates (4 W32 groups a point, pb times
// that many in a row: a multiple of 32, or nearly so, for every d): it loads
// the group (32 bytes, one group ahead), quantizes it, packs the 8 codes
// (aligned to 8 bits) into one 64-bit word and transposes it as an 8 x 8 bit
// matrix, so that byte 7 - l holds bit plane l of the 8 coordinates: byte g of
// the point's plane-l row. The plane rows (W32 words each) are collected in
// shared memory, where the pb points' rows of a plane are adjacent as they are
// in memory, and written out contiguously. One point per warp left half of the
// lanes without a group at d = 64 and a quarter of the rounds at d = 384.
constexpr int QP_THREADS = 256;

// Points per warp: at least four rounds of 32 groups, within 2 KB per warp.
int quantize_points(int W32, int bits) {
  int pb = 1;
  while (pb < 32 && pb * 4 * W32 < 128 && bits * pb * 2 * W32 * 4 <= 2048) pb <<= 1;
  // an odd number of half rounds: one more doubling fills it
  if ((pb * 4 * W32) % 32 != 0 && pb < 32 && bits * pb * 2 * W32 * 4 <= 4096) pb <<= 1;
  return pb;
}

__global__ void __launch_bounds__(QP_THREADS)
quantize_planes_kernel(const float* __restrict__ x, int64_t n, int d, int W32, const float* __restrict__ lo0,
                       const float* __restrict__ scale0, int bits, int vec4, int pb, const uint32_t* __restrict__ seg,
                       uint32_t* __restrict__ planes) {
  extern __shared__ __align__(16) uint32_t qsm[];
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  uint32_t* word_s = qsm + (size_t)wib * bits * pb * W32;  // [bits][pb][W32]
  uint8_t* byte_s = reinterpret_cast<uint8_t*>(word_s);
  const int groups = 4 * W32;
  const int gstep = 32 % groups, pstep = 32 / groups;  // (point, group) of a lane's next item
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const int64_t blocks = (n + pb - 1) / pb;
  for (int64_t b = warp; b < blocks; b += nwarps) {
    const int64_t i0 = b * pb;
    const int np = (int)(n - i0 < pb ? n - i0 : pb);
    float v[8];
    auto load = [&](int pt, int g) {
      const int c0 = 8 * g;
      const float* src = x + (size_t)(i0 + pt) * d + c0;
      if (vec4) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const float4 q = pt < np && c0 + 4 * h < d ? __ldcs(reinterpret_cast<const float4*>(src + 4 * h))
                                                     : make_float4(0.f, 0.f, 0.f, 0.f);
          v[4 * h] = q.x;
          v[4 * h + 1] = q.y;
          v[4 * h + 2] = q.z;
          v[4 * h + 3] = q.w;
        }
      } else {
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = pt < np && c0 + u < d ? __ldg(src + u) : 0.f;
      }
    };
    int pt = lane / groups, g = lane % groups;
    load(pt, g);
    while (pt < np) {
      float q[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) q[u] = v[u];
      const int cpt = pt, cg = g;
      pt += pstep;
      g += gstep;
      if (g >= groups) {
        g -= groups;
        ++pt;
      }
      load(pt, g);
      const int c0 = 8 * cg;
      // segmented rows take their own set's range
      const size_t so = seg ? (size_t)__ldg(seg + i0 + cpt) * d : 0;
      const float* __restrict__ lo = lo0 + so + c0;
      const float* __restrict__ scale = scale0 + so + c0;
      float lov[8], scv[8];
      if (vec4) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const bool in = c0 + 4 * h < d;
          const float4 l = in ? __ldg(reinterpret_cast<const float4*>(lo + 4 * h)) : make_float4(0.f, 0.f, 0.f, 0.f);
          const float4 c = in ? __ldg(reinterpret_cast<const float4*>(scale + 4 * h)) : make_float4(0.f, 0.f, 0.f, 0.f);
          lov[4 * h] = l.x;
          lov[4 * h + 1] = l.y;
          lov[4 * h + 2] = l.z;
          lov[4 * h + 3] = l.w;
          scv[4 * h] = c.x;
          scv[4 * h + 1] = c.y;
          scv[4 * h + 2] = c.z;
          scv[4 * h + 3] = c.w;
        }
      } else {
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          lov[u] = c0 + u < d ? __ldg(lo + u) : 0.f;
          scv[u] = c0 + u < d ? __ldg(scale + u) : 0.f;
        }
      }
      // coordinates past d have scale 0: code 0
      uint32_t w0 = 0, w1 = 0;  // codes of coordinates c0 .. c0+3 and c0+4 .. c0+7, one per byte
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        w0 |= quantize_one(q[u], lov[u], scv[u], bits) << (8 * u);
        w1 |= quantize_one(q[u + 4], lov[u + 4], scv[u + 4], bits) << (8 * u);
      }
      // align every code to 8 bits (the shift stays inside each byte)
      const uint64_t packed = ((uint64_t)w1 << 32 | w0) << (8 - bits);
      const uint64_t tr = transpose8x8(packed);
#pragma unroll
      for (int l = 0; l < 8; ++l)
        if (l < bits) byte_s[(l * pb + cpt) * groups + cg] = (uint8_t)(tr >> (8 * (7 - l)));
    }
    __syncwarp();
    const int words = np * W32;
    for (int l = 0; l < bits; ++l)
      for (int m = lane; m < words; m += 32) planes[((size_t)l * n + i0) * W32 + m] = word_s[l * pb * W32 + m];
    __syncwarp();
  }
}

__global__ void quantize_codes_kernel(const float* __restrict__ x, int64_t total, int d,
                                      const float* __restrict__ lo,
                                      const float* __restrict__ scale, int bits,
                                      uint8_t* __restrict__ codes, int* __restrict__ err) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const float v = x[e];
    if (!isfinite(v)) {
      hf_raise(err, HF_ERRBIT_NONFINITE);
      codes[e] = 0;
      continue;
    }
    const int c = (int)(e % d);
    codes[e] = (uint8_t)quantize_one(v, lo[c], scale[c], bits);
  }
}

__global__ void planes_to_codes_kernel(const uint32_t* __restrict__ planes, int64_t n, int d,
                                       int W32, int bits, uint8_t* __restrict__ codes) {
  const int64_t total = n * d;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = e / d;
    const int c = (int)(e - i * d);
    uint32_t v = 0;
    for (int l = 0; l < bits; ++l)
      v = (v << 1) | ((planes[((size_t)l * n + i) * W32 + (c >> 5)] >> (c & 31)) & 1u);
    codes[e] = (uint8_t)v;
  }
}

// Order-preserving map of floats to unsigned integers (min / max by integer
// atomics; -0 counts as below +0, which leaves every code unchanged).
__device__ __forceinline__ uint32_t float_rank(float v) {
  const uint32_t b = __float_as_uint(v);
  return (b & 0x80000000u) ? ~b : b | 0x80000000u;
}
__device__ __forceinline__ float rank_float(uint32_t r) {
  return __uint_as_float((r & 0x80000000u) ? r & 0x7fffffffu : ~r);
}

// Range of every set of a segmented matrix. Block (row range, column chunk): a
// warp takes 32 / cg rows at a time, cg lanes of VEC consecutive columns each
// (16-byte loads when VEC = 4), four rows per lane in flight; the range's minima
// and maxima are reduced over the block's warps and folded into its set's
// running range (kept as float_rank values in lo / scale) by atomics. The first
// rpb rows of every set are a block's, and every chunk of rpb rows of the matrix
// is another's, for what it holds past the first rpb rows of the set it starts
// in: each block has rows of one set, whatever the sets' sizes. One block per
// set and 32 columns left a 200,000-row set to 8 warps (1.2M x 128 in 23 sets:
// 3.35 ms; the segmented build + graph went from 19.5 to 16.6 ms with an even
// split), and chunks alone, their sets one after the other, took 0.32 ms for 256
// sets of 2 x 16 (SMALL_SETS). Bound by HBM: the points are read once.
constexpr int SR_WARPS = 8;
template <int VEC>
__global__ void __launch_bounds__(SR_WARPS * 32)
seg_range_kernel(const float* __restrict__ x, int64_t n, int d, const int64_t* __restrict__ off, int nseg,
                 const uint32_t* __restrict__ seg, int64_t rpb, int cg, uint32_t* __restrict__ lo,
                 uint32_t* __restrict__ hi, int* __restrict__ err) {
  __shared__ float smn[SR_WARPS][32 * VEC], smx[SR_WARPS][32 * VEC];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int c0 = (int)blockIdx.y * cg * VEC;             // first column of the block
  const int c = c0 + (lane % cg) * VEC, sub = lane / cg;  // this lane's columns and row within the warp's group
  const int rstep = SR_WARPS * (32 / cg);
  // rows [a, b) of one set
  uint32_t set;
  int64_t a, b;
  if ((int)blockIdx.x < nseg) {
    set = blockIdx.x;
    a = __ldg(off + set);
    b = a + rpb;
  } else {
    const int64_t r0 = (int64_t)(blockIdx.x - nseg) * rpb;
    set = __ldg(seg + r0);
    a = __ldg(off + set) + rpb;
    if (a < r0) a = r0;
    b = r0 + rpb;
  }
  const int64_t end = __ldg(off + set + 1);
  if (b > end) b = end;
  if (a >= b) return;
  bool bad = false;
  float mn[VEC], mx[VEC];
#pragma unroll
  for (int v = 0; v < VEC; ++v) {
    mn[v] = INFINITY;
    mx[v] = -INFINITY;
  }
  auto take = [&](const float* q) {
#pragma unroll
    for (int v = 0; v < VEC; ++v) {
      bad |= !isfinite(q[v]);
      mn[v] = fminf(mn[v], q[v]);
      mx[v] = fmaxf(mx[v], q[v]);
    }
  };
  if (c < d) {
    int64_t r = a + warp * (32 / cg) + sub;
    constexpr int UN = 4;
    for (; r + (UN - 1) * rstep < b; r += UN * rstep) {
      float q[UN][VEC];
#pragma unroll
      for (int u = 0; u < UN; ++u) {
        const float* src = x + (size_t)(r + u * rstep) * d + c;
        if (VEC == 4) *reinterpret_cast<float4*>(q[u]) = __ldg(reinterpret_cast<const float4*>(src));
        else q[u][0] = __ldg(src);
      }
#pragma unroll
      for (int u = 0; u < UN; ++u) take(q[u]);
    }
    for (; r < b; r += rstep) {
      float q[VEC];
      const float* src = x + (size_t)r * d + c;
      if (VEC == 4) *reinterpret_cast<float4*>(q) = __ldg(reinterpret_cast<const float4*>(src));
      else q[0] = __ldg(src);
      take(q);
    }
  }
#pragma unroll
  for (int v = 0; v < VEC; ++v) {
    smn[warp][lane * VEC + v] = mn[v];
    smx[warp][lane * VEC + v] = mx[v];
  }
  __syncthreads();
  for (int j = threadIdx.x; j < cg * VEC; j += SR_WARPS * 32) {
    if (c0 + j >= d) break;
    float m0 = INFINITY, m1 = -INFINITY;
    for (int w = 0; w < SR_WARPS; ++w)
      for (int q = j; q < 32 * VEC; q += cg * VEC) {
        m0 = fminf(m0, smn[w][q]);
        m1 = fmaxf(m1, smx[w][q]);
      }
    atomicMin(lo + (size_t)set * d + c0 + j, float_rank(m0));
    atomicMax(hi + (size_t)set * d + c0 + j, float_rank(m1));
  }
  if (bad) hf_raise(err, HF_ERRBIT_NONFINITE);
}

// float_rank ranges -> lo and scale in place, with range_final_kernel's formula.
__global__ void seg_range_final_kernel(int64_t count, int bits, float* __restrict__ lo, float* __restrict__ scale) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= count) return;
  const float mn = rank_float(__float_as_uint(lo[e])), mx = rank_float(__float_as_uint(scale[e]));
  lo[e] = mn;
  const float width = __fsub_rn(mx, mn);
  scale[e] = width > 0.0f ? (float)((double)(1u << bits) / (double)width) : 0.0f;
}

// Set index of every row of a segmented matrix (binary search of the offsets).
__global__ void seg_of_row_kernel(const int64_t* __restrict__ off, int nseg, int64_t n, uint32_t* __restrict__ seg,
                                  uint64_t* __restrict__ seg64) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    int lo = 0, hi = nseg - 1;  // last set whose offset is <= i
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (__ldg(off + mid) <= i) lo = mid;
      else hi = mid - 1;
    }
    seg[i] = (uint32_t)lo;
    if (seg64) seg64[i] = (uint64_t)lo;
  }
}

int64_t range_threads(int64_t n, int d, int vec) {
  const int64_t groups = d / vec;
  int64_t target = 152 * 2048;
  int64_t reps = (target + groups - 1) / groups;
  // eight rows per thread at least: with one, a 20,000 x 16 matrix's partials
  // were as large as the matrix (final reduction 17.7 us)
  const int64_t rows_max = (n + 7) / 8;
  if (reps > rows_max) reps = rows_max;
  if (reps < 1) reps = 1;
  return reps * groups;
}

}  // namespace

size_t range_scratch_bytes(int64_t n, int d) {
  const int vec = (d % 4 == 0) ? 4 : 1;
  return (size_t)range_threads(n, d, vec) * vec * 2 * sizeof(float);
}

void launch_range(const float* x, int64_t n, int d, float* lo, float* scale, int bits, int* err,
                  void* scratch, size_t scratch_bytes, cudaStream_t s) {
  const bool v4 = (d % 4 == 0) && ((reinterpret_cast<uintptr_t>(x) & 15) == 0);
  const int vec = v4 ? 4 : 1;
  int64_t nthreads = range_threads(n, d, (d % 4 == 0) ? 4 : 1);
  if (!v4) nthreads = range_threads(n, d, 1);
  float* pmin = static_cast<float*>(scratch);
  float* pmax = pmin + nthreads * vec;
  (void)scratch_bytes;
  const int64_t total_vec = n * d / vec;
  const unsigned blocks = hf_blocks(nthreads, RANGE_THREADS);
  if (v4)
    range_partial_kernel<4><<<blocks, RANGE_THREADS, 0, s>>>(x, total_vec, d, nthreads, pmin, pmax, err);
  else
    range_partial_kernel<1><<<blocks, RANGE_THREADS, 0, s>>>(x, total_vec, d, nthreads, pmin, pmax, err);
  hf_after_launch("range_partial_kernel", s);
  range_final_kernel<<<d, 256, 0, s>>>(pmin, pmax, nthreads, vec, d, bits, lo, scale);
  hf_after_launch("range_final_kernel", s);
}

void launch_seg_range(const float* x, int64_t n, int d, const int64_t* off, const uint32_t* seg, int nseg, int bits,
                      float* lo, float* scale, int* err, cudaStream_t s) {
  const int64_t count = (int64_t)nseg * d;
  uint32_t* ulo = reinterpret_cast<uint32_t*>(lo);
  uint32_t* uhi = reinterpret_cast<uint32_t*>(scale);
  cudaMemsetAsync(ulo, 0xff, (size_t)count * 4, s);
  cudaMemsetAsync(uhi, 0, (size_t)count * 4, s);
  const bool v4 = d % 4 == 0 && (reinterpret_cast<uintptr_t>(x) & 15) == 0;
  const int groups = v4 ? d / 4 : d;
  int cg = 1;
  while (cg < 32 && cg < groups) cg <<= 1;
  const int ychunks = (groups + cg - 1) / cg;
  // about 8 blocks per SM, at least 4 rows per lane
  int64_t rpb = (n * ychunks + 152 * 8 - 1) / (152 * 8);
  const int64_t least = (int64_t)SR_WARPS * (32 / cg) * 4;
  if (rpb < least) rpb = least;
  const dim3 grid((unsigned)nseg + hf_blocks(n, (int)rpb), (unsigned)ychunks);
  if (v4)
    seg_range_kernel<4><<<grid, SR_WARPS * 32, 0, s>>>(x, n, d, off, nseg, seg, rpb, cg, ulo, uhi, err);
  else
    seg_range_kernel<1><<<grid, SR_WARPS * 32, 0, s>>>(x, n, d, off, nseg, seg, rpb, cg, ulo, uhi, err);
  hf_after_launch("seg_range_kernel", s);
  seg_range_final_kernel<<<hf_blocks(count, 256), 256, 0, s>>>(count, bits, lo, scale);
  hf_after_launch("seg_range_final_kernel", s);
}

void launch_seg_of_row(const int64_t* off, int nseg, int64_t n, uint32_t* seg, uint64_t* seg64, cudaStream_t s) {
  seg_of_row_kernel<<<hf_blocks(n, 256, 152 * 8), 256, 0, s>>>(off, nseg, n, seg, seg64);
  hf_after_launch("seg_of_row_kernel", s);
}

void launch_quantize_planes(const float* x, int64_t n, int d, const float* lo, const float* scale,
                            int bits, uint32_t* planes, int* err, cudaStream_t s, const uint32_t* seg) {
  (void)err;
  const int W32 = (d + 31) / 32;
  const int vec4 = d % 4 == 0 && (reinterpret_cast<uintptr_t>(x) & 15) == 0;
  const int pb = quantize_points(W32, bits);
  const size_t smem = (size_t)(QP_THREADS / 32) * bits * pb * W32 * 4;
  if (smem > 48 * 1024)
    cudaFuncSetAttribute((const void*)quantize_planes_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  quantize_planes_kernel<<<hf_blocks((n + pb - 1) / pb * 32, QP_THREADS, 152 * 16), QP_THREADS, smem, s>>>(
      x, n, d, W32, lo, scale, bits, vec4, pb, seg, planes);
  hf_after_launch("quantize_planes_kernel", s);
}

void launch_quantize_codes(const float* x, int64_t n, int d, const float* lo, const float* scale,
                           int bits, uint8_t* codes, int* err, cudaStream_t s) {
  const int64_t total = n * d;
  quantize_codes_kernel<<<hf_blocks(total, 256, 152 * 16), 256, 0, s>>>(x, total, d, lo, scale, bits,
                                                                       codes, err); hf_after_launch("quantize_codes_kernel", s);
}

void launch_planes_to_codes(const uint32_t* planes, int64_t n, int d, int bits, uint8_t* codes,
                            cudaStream_t s) {
  const int W32 = (d + 31) / 32;
  planes_to_codes_kernel<<<hf_blocks(n * d, 256, 152 * 16), 256, 0, s>>>(planes, n, d, W32, bits, codes); hf_after_launch("planes_to_codes_kernel", s);
}
