// Window distances and top-k merge (plain float32 form).
//
// Paper, Algorithm 2: in every sort, the points lying a few places before and
// after a point in that sort's Hilbert order join its candidates, and the
// best k candidates by vector distance are the result. Here the window is w
// positions on each side, the distance is the float32 squared Euclidean
// distance with exact coordinate differences, and each point's list (k pairs
// of (distance, index), ascending) is merged tree by tree, so the candidate
// set is never materialised beyond one tree.
//
// Two kernels per tree:
//   pair_kernel   the distances of the pairs (p, p + delta), 1 <= delta <= w,
//                 each computed once, into a band D[delta - 1][p];
//   merge_kernel  each point's 2w band entries (its right ones in column p,
//                 its left ones, the pairs (p - delta, p), in column
//                 p - delta) into its list.
// The band goes through memory between them, in row chunks of at most
// BAND_BYTES: 8 w bytes a point written and read against 2 w d lane operations
// (w = 32, d = 384: 0.2 ms of traffic per 3M-point tree beside 2.4 ms of
// arithmetic at the pipe's rate). One kernel that did both had to own its
// points on both sides: a block of 512 rows recomputed the rows of every left
// neighbour (up to 1.4 times the pairs at w = 250), and half of its threads
// merged, from shared memory with 32-way bank conflicts, while the FP32 pipe
// idled. Per 3M x 384 tree at w = 32: 5.8 ms in that form, 3.2 + 0.43 ms here;
// build + graph 3M x 384, T = 32, w = 32: 202.9 -> 144.0 ms; 100,003 x 100,
// T = 8, w = 250: 11.9 -> 4.5 ms.
//
// (x_p - x_q)^2 and (x_q - x_p)^2 are equal and the coordinates are always
// summed in order, so a pair scores the same in every tree.
#include <cuda_runtime.h>
#include <math.h>

#include "hf_internal.cuh"
#include "topk_list.cuh"

namespace {

constexpr int DC = 16;          // coordinates per staged chunk
constexpr int UR = 8;           // rows per unit
constexpr int UC = 8;           // offsets per unit
constexpr int kSms = 152;
// Memory of one chunk's band.
constexpr size_t BAND_BYTES = (size_t)256 << 20;

__device__ __forceinline__ void cp_async4(uint32_t dst, const float* src, bool valid) {
  const int sz = valid ? 4 : 0;  // 0: zero-fill, nothing read
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(sz) : "memory");
}
__device__ __forceinline__ void cp_async16(uint32_t dst, const float* src, bool valid) {
  const int sz = valid ? 16 : 0;
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(sz) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_1() { asm volatile("cp.async.wait_group 1;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_0() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

// Byte offset of 16-byte piece q (coordinates 4q .. 4q+3 of the chunk) of
// staged row r: two rows per 128-byte line, the line's eight pieces permuted
// by the row's group of 8, so that the rows 8 apart that a warp reads together
// fall in different banks.
__device__ __forceinline__ uint32_t piece_off(int r, int q) {
  return (uint32_t)((r >> 1) * 128 + (((((r & 1) << 2) | q) ^ ((r >> 3) & 7)) << 4));
}

// Stage coordinates [c0, c0 + DC) of staged rows [0, NR): 16 bytes a copy when
// rows are 16-byte aligned (VEC), else 4.
template <int NT, bool VEC>
__device__ __forceinline__ void stage_chunk(uint32_t buf, int NR, const uint32_t* srow, const float* __restrict__ x,
                                            int d, int c0) {
  if (VEC) {
    const int q = threadIdx.x & 3;
    const bool in = c0 + 4 * q < d;
    const float* xc = x + c0 + 4 * q;
    for (int r = threadIdx.x >> 2; r < NR; r += NT / 4) {
      const uint32_t pid = srow[r];
      const bool ok = in && pid != 0xffffffffu;
      cp_async16(buf + piece_off(r, q), ok ? xc + (size_t)pid * d : x, ok);
    }
  } else {
    const int c = threadIdx.x & (DC - 1);
    const bool in = c0 + c < d;
    const float* xc = x + c0 + c;
    for (int r = threadIdx.x / DC; r < NR; r += NT / DC) {
      const uint32_t pid = srow[r];
      const bool ok = in && pid != 0xffffffffu;
      cp_async4(buf + piece_off(r, c >> 2) + (c & 3) * 4, ok ? xc + (size_t)pid * d : x, ok);
    }
  }
}

// Tile shape of a launch: NT threads, OG offset groups of 8 -> NT / OG row
// groups of 8.
__host__ __device__ constexpr int tile_rows(int nt, int og) { return nt / og * UR; }

struct PairArgs {
  const float* x;
  const uint32_t* sigma;
  int64_t n, row0;  // D's column 0 is position row0
  int64_t pitch;    // columns of D (a multiple of the tile rows)
  int d, w;
  int dlo0;         // first offset of the launch; blockIdx.y adds 8 OG each
  float* D;         // [w][pitch]
};

// Staged rows: the tile's R rows and the R + 8 OG rows from dlo - 1 on; one
// range while they touch, else two.
__host__ __device__ __forceinline__ int staged_rows(int R, int OT, int dlo) {
  return (dlo - 1 < R ? dlo - 1 : R) + R + OT;
}

// Distances of the pairs (p, p + delta): R = tile_rows positions times 8 OG
// offsets per block, an 8-row x 8-offset unit (64 sums in registers) per
// thread. The rows are staged 16 coordinates at a time, double-buffered
// against the arithmetic, and read four coordinates of a row at a time: a
// thread holds its 8 own rows' piece and streams the 15 rows its offsets
// reach, each pair adding its coordinates in order. HAM: the rows are binary
// sketches (d 32-bit words each) and the distance is their Hamming distance
// (the paper's second-stage filter).
// Bound by the FP32 pipe (POPC for HAM): 2 lane operations per pair and
// coordinate; a loop of nothing else reaches 32 T/s on this chip, packed pair
// instructions the same; this kernel 23 T/s (3M x 384, w = 32), 80 % of its
// instructions the arithmetic. Coordinate-major staging by 4-byte copies put
// 43 % of them elsewhere (17 T/s).
template <int NT, int OG, bool HAM, bool VEC>
__global__ void __launch_bounds__(NT, 512 / NT) pair_kernel(const PairArgs a) {
  constexpr int R = tile_rows(NT, OG), OT = OG * UC;
  extern __shared__ __align__(128) unsigned char smem[];
  const int dlo = a.dlo0 + (int)blockIdx.y * OT;
  const int64_t s = a.row0 + (int64_t)blockIdx.x * R;
  if (s + dlo >= a.n) return;  // no pair of this tile exists
  const int bofs = dlo - 1 < R ? dlo - 1 : R;  // staged row of position s + dlo - 1
  const int NR = bofs + R + OT;                // a multiple of 16
  const uint32_t buf0 = (uint32_t)__cvta_generic_to_shared(smem);
  const uint32_t buf1 = buf0 + (uint32_t)NR * 64;
  uint32_t* srow = reinterpret_cast<uint32_t*>(smem + (size_t)NR * 128);
  for (int r = threadIdx.x; r < NR; r += NT) {
    const int64_t p = s + (r < bofs ? r : r - bofs + dlo - 1);
    srow[r] = p < a.n ? __ldg(a.sigma + p) : 0xffffffffu;
  }
  __syncthreads();

  // unit of this thread: rows pr .. pr+7, offsets dlo + 8o .. dlo + 8o + 7
  const int g = threadIdx.x / OG, o = threadIdx.x % OG;
  const int pr = UR * g;
  const int br = bofs + pr + UC * o;  // staged row of offset -1 of row 0 (a multiple of 8)
  const uint32_t ao = piece_off(pr, 0), bo0 = piece_off(br, 0), bo1 = piece_off(br + 8, 0);

  float acc[UR][UC];
#pragma unroll
  for (int t = 0; t < UR; ++t)
#pragma unroll
    for (int c = 0; c < UC; ++c) acc[t][c] = 0.f;

  const int nchunks = (a.d + DC - 1) / DC;
  stage_chunk<NT, VEC>(buf0, NR, srow, a.x, a.d, 0);
  cp_async_commit();
  for (int ch = 0; ch < nchunks; ++ch) {
    const uint32_t cur = (ch & 1) ? buf1 : buf0, nxt = (ch & 1) ? buf0 : buf1;
    if (ch + 1 < nchunks) stage_chunk<NT, VEC>(nxt, NR, srow, a.x, a.d, (ch + 1) * DC);
    cp_async_commit();
    cp_async_wait_1();
    __syncthreads();
    const unsigned char* cb = smem + (cur - buf0);
    // the last chunk holds what is left of d (its padding adds exact zeros)
    const int left = a.d - ch * DC, nq = left < DC ? (left + 3) >> 2 : DC / 4;
#pragma unroll 1
    for (int q = 0; q < nq; ++q) {
      // row t of a group of 8 lies (t / 2) lines on, its piece index XORed
      // with 4 for odd t
      float4 av[UR];
#pragma unroll
      for (int t = 0; t < UR; ++t)
        av[t] = *reinterpret_cast<const float4*>(cb + ((ao ^ (uint32_t)((((t & 1) << 2) | 0) << 4)) ^ (uint32_t)(q << 4)) +
                                                 (t >> 1) * 128);
#pragma unroll
      for (int j = 1; j < 16; ++j) {  // b row: t + c = j - 1
        const uint32_t bo = j < 8 ? bo0 : bo1;
        const float4 bv = *reinterpret_cast<const float4*>(cb + ((bo ^ (uint32_t)((j & 1) << 6)) ^ (uint32_t)(q << 4)) +
                                                           ((j & 7) >> 1) * 128);
#pragma unroll
        for (int t = 0; t < UR; ++t) {
          const int c = j - 1 - t;
          if (c < 0 || c >= UC) continue;
          if (HAM) {
            // integer popcount sums kept in the float registers' bits
            uint32_t u = __float_as_uint(acc[t][c]);
            u += (uint32_t)__popc(__float_as_uint(av[t].x) ^ __float_as_uint(bv.x));
            u += (uint32_t)__popc(__float_as_uint(av[t].y) ^ __float_as_uint(bv.y));
            u += (uint32_t)__popc(__float_as_uint(av[t].z) ^ __float_as_uint(bv.z));
            u += (uint32_t)__popc(__float_as_uint(av[t].w) ^ __float_as_uint(bv.w));
            acc[t][c] = __uint_as_float(u);
          } else {
            float e = av[t].x - bv.x;
            float v = fmaf(e, e, acc[t][c]);
            e = av[t].y - bv.y;
            v = fmaf(e, e, v);
            e = av[t].z - bv.z;
            v = fmaf(e, e, v);
            e = av[t].w - bv.w;
            acc[t][c] = fmaf(e, e, v);
          }
        }
      }
    }
    __syncthreads();
  }
  cp_async_wait_0();

  float* out = a.D + (s - a.row0) + pr;
#pragma unroll
  for (int c = 0; c < UC; ++c) {
    const int delta = dlo + UC * o + c;
    if (delta <= a.w) {
      float* row = out + (size_t)(delta - 1) * a.pitch;
#pragma unroll
      for (int t = 0; t < UR; t += 4) {
        float4 v = make_float4(acc[t][c], acc[t + 1][c], acc[t + 2][c], acc[t + 3][c]);
        if (HAM)
          v = make_float4((float)__float_as_uint(v.x), (float)__float_as_uint(v.y), (float)__float_as_uint(v.z),
                          (float)__float_as_uint(v.w));
        *reinterpret_cast<float4*>(row + t) = v;
      }
    }
  }
}

struct MergeArgs {
  const float* D;
  const uint32_t* sigma;
  int64_t n, row0, pitch;
  int64_t p0, p1;  // points of this launch
  int w;
  uint32_t* lidx;
  float* ldist;
  const uint32_t* segr;    // segmented forest: set of each point, or null
  const int64_t* segoff;
};

// One thread per position, its point's list in registers. 32 offsets at a
// time, a thread first marks the right and left entries that its list's last
// distance does not exclude (the lanes of a warp read consecutive columns of
// the band), then inserts its marked ones; the lanes insert their own
// candidates side by side, so a warp makes as many insertion steps as its
// busiest lane has marks (about ten on settled lists) where a lane-by-lane
// scan made one for nearly every offset. Bound by the band's trip through
// memory and, while the lists fill, by the insertions.
template <int KP>
__global__ void __launch_bounds__(128) merge_kernel(const MergeArgs a) {
  const int64_t p = a.p0 + (int64_t)blockIdx.x * 128 + threadIdx.x;
  if (p >= a.p1) return;
  const uint32_t ip = __ldg(a.sigma + p);
  // offsets this point may take on each side (its set's block of the order)
  int64_t plo = 0, phi = a.n;
  if (a.segr) {
    const uint32_t sg = __ldg(a.segr + ip);
    plo = __ldg(a.segoff + sg);
    phi = __ldg(a.segoff + sg + 1);
  }
  const int rmax = (int)(phi - 1 - p < a.w ? phi - 1 - p : a.w);
  const int lmax = (int)(p - plo < a.w ? p - plo : a.w);
  ListK<KP> L;
  L.load(a.ldist + (size_t)ip * KP, a.lidx + (size_t)ip * KP);
  bool changed = false;
  const float* col = a.D + (p - a.row0);
  const size_t pitch = a.pitch;
  for (int d0 = 1; d0 <= a.w; d0 += 32) {
    uint32_t mr = 0, ml = 0;
    const float last = L.d[KP - 1];
    const float* row = col + (size_t)(d0 - 1) * pitch;
#pragma unroll
    for (int j0 = 0; j0 < 32; j0 += 8) {
      float vr[8], vl[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int delta = d0 + j0 + j;
        vr[j] = delta <= rmax ? __ldg(row + (size_t)(j0 + j) * pitch) : NAN;
        vl[j] = delta <= lmax ? __ldg(row + (size_t)(j0 + j) * pitch - delta) : NAN;
      }
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        if (vr[j] <= last) mr |= 1u << (j0 + j);
        if (vl[j] <= last) ml |= 1u << (j0 + j);
      }
    }
    // the next marked candidate is on its way while this one is inserted
    float nv = NAN;
    uint32_t nid = 0xffffffffu;
    auto next = [&]() {
      const bool right = mr != 0;
      const uint32_t m = right ? mr : ml;
      nv = NAN;
      if (!m) return;
      const int j = __ffs(m) - 1;
      if (right) mr &= mr - 1;
      else ml &= ml - 1;
      const int delta = d0 + j;
      nv = __ldg(row + (size_t)j * pitch - (right ? 0 : delta));
      nid = __ldg(a.sigma + (right ? p + delta : p - delta));
    };
    bool more = (mr | ml) != 0;
    changed |= more;
    next();
    while (more) {
      const float v = nv;
      const uint32_t id = nid;
      more = (mr | ml) != 0;
      next();
      L.offer(v, id);
    }
  }
  if (changed) L.store(a.ldist + (size_t)ip * KP, a.lidx + (size_t)ip * KP);
}

__global__ void list_init_kernel(uint32_t* __restrict__ idx, float* __restrict__ dist, int64_t count) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < count;
       e += (int64_t)gridDim.x * blockDim.x) {
    idx[e] = 0xffffffffu;
    dist[e] = INFINITY;
  }
}

// Row chunk of a tree: `rows` points per chunk, the band's column pitch.
struct BandGeom {
  int64_t rows, pitch;
};
BandGeom band_geom(int64_t n, int w) {
  BandGeom g;
  const int64_t most = (int64_t)(BAND_BYTES / 4) / w;  // columns that fit, 90,000 at the widest window
  // chunk + left halo (w columns) + tile rounding
  const int64_t usable = most - w - 2 * 1024;
  const int64_t chunks = (n + usable - 1) / usable;
  g.rows = (n + chunks - 1) / chunks;
  g.pitch = (g.rows + (chunks > 1 ? w : 0) + 1024 + 1023) / 1024 * 1024;
  return g;
}

template <int NT, int OG, bool HAM>
int launch_pairs(PairArgs a, int dlo, int ytiles, int64_t cols, cudaStream_t s) {
  constexpr int R = tile_rows(NT, OG), OT = OG * UC;
  int nr = 0;
  for (int y = 0; y < ytiles; ++y) {
    const int v = staged_rows(R, OT, dlo + y * OT);
    if (v > nr) nr = v;
  }
  const size_t smem = (size_t)nr * (128 + 4);
  const bool vec = a.d % 4 == 0 && (reinterpret_cast<uintptr_t>(a.x) & 15) == 0;
  const void* fn = vec ? (const void*)pair_kernel<NT, OG, HAM, true> : (const void*)pair_kernel<NT, OG, HAM, false>;
  if (cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess) return HF_ECUDA;
  a.dlo0 = dlo;
  const dim3 grid(hf_blocks(cols, R), (unsigned)ytiles);
  if (vec)
    pair_kernel<NT, OG, HAM, true><<<grid, NT, smem, s>>>(a);
  else
    pair_kernel<NT, OG, HAM, false><<<grid, NT, smem, s>>>(a);
  hf_after_launch(HAM ? "pair_kernel<hamming>" : "pair_kernel", s);
  return HF_OK;
}

// Offsets 1 .. w in tiles of 64 (256 rows; the fewest staged rows per pair),
// the rest in tiles of 32 (512 rows) and 16 (512 rows of 128 threads), so that
// at most 15 offsets are computed beyond w. A launch that leaves SMs idle lasts
// as long as one block, and rows that are not 16-byte aligned are staged in 4-byte
// copies, fewer per thread in the tiles of 64: they take such a launch's rest too
// (200 x 33, T = 8, w = 2: 0.30 -> 0.24 ms the graph; aligned rows are bound by
// the arithmetic, which the wider tile has more of: 200 x 384: 0.75 -> 0.86).
// nt = 512, for plans that ask for it (the tuner tries both): 64-offset tiles of
// 512 rows, one block per SM; at windows from 64 to 704 between 3 % faster
// (20,000 x 384, w = 128) and 12 % slower (100,003 x 100, w = 64) than nt = 256,
// 50 % on 20,000 x 384 at w = 64.
template <bool HAM>
int launch_band(const PairArgs& a, int64_t cols, int nt, cudaStream_t s) {
  int full = a.w / 64, rest = a.w % 64;
  const bool vec = a.d % 4 == 0 && (reinterpret_cast<uintptr_t>(a.x) & 15) == 0;
  if (rest > 48 || (rest > 0 && !vec && nt != 512 && (cols + 255) / 256 * (full + 1) <= kSms)) {
    ++full;
    rest = 0;
  }
  int rc = HF_OK;
  if (full) rc = nt == 512 ? launch_pairs<512, 8, HAM>(a, 1, full, cols, s) : launch_pairs<256, 8, HAM>(a, 1, full, cols, s);
  int dlo = 64 * full + 1;
  if (rc == HF_OK && rest > 16) {
    rc = launch_pairs<256, 4, HAM>(a, dlo, 1, cols, s);
    dlo += 32;
    rest -= 32;
  }
  if (rc == HF_OK && rest > 0) rc = launch_pairs<128, 2, HAM>(a, dlo, 1, cols, s);
  return rc;
}

template <int KP>
void launch_merge(const MergeArgs& a, cudaStream_t s) {
  merge_kernel<KP><<<hf_blocks(a.p1 - a.p0, 128), 128, 0, s>>>(a);
  hf_after_launch("merge_kernel", s);
}

template <bool HAM>
int launch_tree(const float* x, int64_t n, int d, const uint32_t* sigma, int w, int kp, uint32_t* li, float* ldd,
                float* band, cudaStream_t s, const uint32_t* segr, const int64_t* segoff, int nt) {
  if (kp != 16 && kp != 32 && kp != 64) return HF_EINVAL;
  const BandGeom g = band_geom(n, w);
  for (int64_t c0 = 0; c0 < n; c0 += g.rows) {
    const int64_t c1 = c0 + g.rows < n ? c0 + g.rows : n;
    const int64_t row0 = c0 > w ? (c0 - w) & ~(int64_t)7 : 0;
    PairArgs pa{x, sigma, n, row0, g.pitch, d, w, 1, band};
    const int rc = launch_band<HAM>(pa, c1 - row0, nt, s);
    if (rc != HF_OK) return rc;
    MergeArgs ma{band, sigma, n, row0, g.pitch, c0, c1, w, li, ldd, segr, segoff};
    switch (kp) {
      case 16: launch_merge<16>(ma, s); break;
      case 32: launch_merge<32>(ma, s); break;
      default: launch_merge<64>(ma, s); break;
    }
  }
  return HF_OK;
}

}  // namespace

void launch_list_init(uint32_t* idx, float* dist, int64_t count, cudaStream_t s) {
  list_init_kernel<<<hf_blocks(count, 256, 152 * 8), 256, 0, s>>>(idx, dist, count);
  hf_after_launch("list_init_kernel", s);
}

int window_list_pitch(int k) { return k <= 16 ? 16 : (k <= 32 ? 32 : 64); }

size_t window_band_bytes(int64_t n, int w) { return (size_t)band_geom(n, w).pitch * w * 4; }

size_t window_band_bytes_most(int64_t n) {
  size_t most = 0;
  for (int w = 1; w <= HF_PLAIN_MAX_W; ++w) {
    const size_t b = window_band_bytes(n, w);
    if (b > most) most = b;
  }
  return most;
}

// w up to HF_PLAIN_MAX_W. Lists have window_list_pitch(k) slots per point;
// band: window_band_bytes(n, w) of scratch.
int launch_window_graph(const float* x, int64_t n, int d, const uint32_t* sigma, int w, int kp,
                        uint32_t* list_idx, float* list_dist, float* band, cudaStream_t s, const uint32_t* segr,
                        const int64_t* segoff, int nt) {
  if (nt != 0 && nt != 256 && nt != 512) return HF_EINVAL;
  return launch_tree<false>(x, n, d, sigma, w, kp, list_idx, list_dist, band, s, segr, segoff, nt);
}

int launch_window_hamming(const uint32_t* sketch, int64_t n, int words, const uint32_t* sigma, int w, int kp,
                          uint32_t* list_idx, float* list_dist, float* band, cudaStream_t s, const uint32_t* segr,
                          const int64_t* segoff) {
  // staged as raw 32-bit words
  return launch_tree<true>(reinterpret_cast<const float*>(sketch), n, words, sigma, w, kp, list_idx, list_dist, band, s,
                           segr, segoff, 0);
}
