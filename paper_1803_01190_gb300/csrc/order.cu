// Spatial (Morton, Z-curve) ordering of the particles before the force sum.
//
// The mixed kernel evaluates Eq. 2 in binary32 on coordinates re-centred on
// an anchor per j-tile: x_j - c and x_i - c are each rounded once to binary32,
// so a pair's difference carries an error of about 2^-24 |x - c|.  For a
// close pair (|d| near the softening) that is a relative error of
// 2^-24 |x - c| / |d|, and with particles in input order a tile spans the
// whole system, |x - c| ~ its radius.  Sorting the particles along a
// space-filling curve first makes every tile of consecutive particles
// spatially compact, so |x - c| is the tile's own size wherever a pair is
// close, and the binary32 coordinates keep their digits.
//
// The order is a deterministic function of the positions alone: the bounding
// box is an exact min/max (order independent), the key of a particle is the
// bit interleave of its three 21-bit cell indices in that box, and the sort is
// stable on (key, input index), so equal keys keep input order.  Results
// therefore stay bit-reproducible (a resumed run recomputes the same order from
// the same positions).
//
// Steps (one force evaluation): bbox partials -> keys -> sort -> gather of the
// positions into sorted order; the epilogue kernels read the sorted partial
// sums through the permutation.  Up to kRankMax particles the sort is two
// launches: every block of 256 sorts its own keys (bitonic, lane shuffles
// below strides of 32), then every particle finds its place by counting the
// smaller keys of each other chunk (binary searches in L2, independent of one
// another) and gathers its position there.  Latency is all it costs at these
// sizes: at N = 2048 the order takes 15 us of kernels (box 3, chunks 6, places
// 5.5) where the dozen launches of the radix sort took about 45; a whole mixed
// evaluation with its copies falls from 202 to 84 us at N = 4096, 336 to 204 at
// 16387, 2088 to 1905 at 65536.  Chunks of 512 measure the same within 3 %.
// Above, the radix sort moves fewer bytes than n / 256 searches per particle.
#include <cuda_runtime.h>

#include <algorithm>

#include <cub/device/device_radix_sort.cuh>

#include "nbody_internal.cuh"

namespace nb {

namespace {

constexpr int kBT = 256;
constexpr int kBboxBlocks = 256;  // partial boxes reduced by one block afterwards
constexpr int kCellBits = 21;     // per coordinate; 63-bit keys
constexpr int kChunk = 256;       // particles sorted by one block
constexpr int kRankWarps = 8;
constexpr int64_t kRankMax = 65536;

// Binary64 as an unsigned integer of the same order, and back.  Minima and
// maxima are integer reductions: an FP64 comparison takes as long as 32 of
// them.
__device__ __forceinline__ uint64_t ordered(double x) {
  const int64_t b = __double_as_longlong(x);
  return (uint64_t)(b ^ ((b >> 63) | (int64_t)0x8000000000000000ull));
}
__device__ __forceinline__ double unordered(uint64_t k) {
  const int64_t b = (int64_t)k;
  return __longlong_as_double(b ^ (~(b >> 63) | (int64_t)0x8000000000000000ull));
}
// over the lanes of a warp: the high words first, then the low words of those
// that hold the winning one
template <bool MAX>
__device__ __forceinline__ uint64_t warp_extreme(uint64_t k) {
  const unsigned h = (unsigned)(k >> 32), l = (unsigned)k, F = 0xFFFFFFFFu;
  const unsigned wh = MAX ? __reduce_max_sync(F, h) : __reduce_min_sync(F, h);
  const unsigned mine = h == wh ? l : MAX ? 0u : F;
  const unsigned wl = MAX ? __reduce_max_sync(F, mine) : __reduce_min_sync(F, mine);
  return ((uint64_t)wh << 32) | wl;
}

// Bounding box of a grid-stride share of [0, n) per block: part[0..2] minima,
// part[3..5] maxima, as ordered integers.  NaNs are left out.
__global__ void __launch_bounds__(kBT) k_bbox_partial(const d4 *__restrict__ posm, int64_t n,
                                                      uint64_t *__restrict__ part) {
  chain_begin();
  __shared__ uint64_t s[6][kBT / 32];
  uint64_t v[6];
#pragma unroll
  for (int c = 0; c < 6; c++) v[c] = ordered(c < 3 ? INFINITY : -INFINITY);
  for (int64_t i = blockIdx.x * (int64_t)kBT + threadIdx.x; i < n; i += (int64_t)gridDim.x * kBT) {
    const d4 p = posm[i];
    const double x[3] = {p.x, p.y, p.z};
#pragma unroll
    for (int c = 0; c < 3; c++) {
      const uint64_t k = ordered(x[c]);
      if (((unsigned)__double2hiint(x[c]) & 0x7FFFFFFFu) <= 0x7FF00000u) {
        v[c] = min(v[c], k);
        v[3 + c] = max(v[3 + c], k);
      }
    }
  }
#pragma unroll
  for (int c = 0; c < 6; c++) {
    v[c] = c < 3 ? warp_extreme<false>(v[c]) : warp_extreme<true>(v[c]);
    if ((threadIdx.x & 31) == 0) s[c][threadIdx.x >> 5] = v[c];
  }
  __syncthreads();
  if (threadIdx.x < 6) {
    const int c = threadIdx.x;
    uint64_t x = s[c][0];
#pragma unroll
    for (int w = 1; w < kBT / 32; w++) x = c < 3 ? min(x, s[c][w]) : max(x, s[c][w]);
    part[blockIdx.x * 6 + c] = x;
  }
}

// Spread the low 21 bits of v to every third bit of a 64-bit word.
__device__ __forceinline__ uint64_t spread3(uint64_t v) {
  v &= 0x1fffffull;
  v = (v | (v << 32)) & 0x1f00000000ffffull;
  v = (v | (v << 16)) & 0x1f0000ff0000ffull;
  v = (v | (v << 8)) & 0x100f00f00f00f00full;
  v = (v | (v << 4)) & 0x10c30c30c30c30c3ull;
  v = (v | (v << 2)) & 0x1249249249249249ull;
  return v;
}

// Cells of the order: (x - lo) * scale, 2^21 - 1 of them across the largest extent.
struct Cells {
  double lo[3], scale;
};

// The cells of the partial boxes' union, by the first six warps of a block.
__device__ __forceinline__ Cells reduce_box(const uint64_t *__restrict__ part, int nparts) {
  __shared__ double box[6];
  const int c = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (c < 6) {
    uint64_t v = part[c];
    for (int b = lane; b < nparts; b += 32)
      v = c < 3 ? min(v, part[b * 6 + c]) : max(v, part[b * 6 + c]);
    v = c < 3 ? warp_extreme<false>(v) : warp_extreme<true>(v);
    if (lane == 0) box[c] = unordered(v);
  }
  __syncthreads();
  Cells q;
  const double span = fmax(fmax(box[3] - box[0], box[4] - box[1]), box[5] - box[2]);
  const double cells = (double)((1u << kCellBits) - 1);
  q.scale = span > 0 ? cells / span : 0.0;
#pragma unroll
  for (int k = 0; k < 3; k++) q.lo[k] = box[k];
  return q;
}

// Morton key of a position (a NaN coordinate lies in cell 0).
__device__ __forceinline__ uint64_t morton_key(const d4 &p, const Cells &q) {
  const double x[3] = {p.x, p.y, p.z};
  uint64_t key = 0;
#pragma unroll
  for (int c = 0; c < 3; c++) {
    const double f = (x[c] - q.lo[c]) * q.scale;
    const bool number = ((unsigned)__double2hiint(f) & 0x7FFFFFFFu) <= 0x7FF00000u;
    const unsigned cell = number ? min(__double2uint_rd(f), (1u << kCellBits) - 1) : 0u;
    key |= spread3(cell) << c;
  }
  return key;
}

__global__ void __launch_bounds__(kBT) k_morton_keys(const d4 *__restrict__ posm, int64_t n,
                                                     const uint64_t *__restrict__ part, int nparts,
                                                     uint64_t *__restrict__ keys,
                                                     int32_t *__restrict__ idx) {
  const Cells q = reduce_box(part, nparts);
  for (int64_t i = blockIdx.x * (int64_t)kBT + threadIdx.x; i < n; i += (int64_t)gridDim.x * kBT) {
    keys[i] = morton_key(posm[i], q);
    idx[i] = (int32_t)i;
  }
}

// Keys of one chunk of kChunk particles, sorted (equal keys in input order);
// the tail of the last chunk is filled with keys above every real one.
__global__ void __launch_bounds__(kChunk) k_sort_chunk(const d4 *__restrict__ posm, int64_t n,
                                                       const uint64_t *__restrict__ part, int nparts,
                                                       uint64_t *__restrict__ keys,
                                                       int32_t *__restrict__ idx) {
  chain_begin();
  __shared__ uint64_t sk[2][kChunk];
  __shared__ int si[2][kChunk];
  const Cells q = reduce_box(part, nparts);
  const int tid = threadIdx.x;
  const int64_t g = blockIdx.x * (int64_t)kChunk + tid;
  uint64_t key = g < n ? morton_key(posm[g], q) : ~(uint64_t)0;
  int id = tid, buf = 0;
  for (int k = 2; k <= kChunk; k <<= 1)
    for (int j = k >> 1; j > 0; j >>= 1) {
      uint64_t okey;
      int oid;
      if (j >= 32) {
        sk[buf][tid] = key;
        si[buf][tid] = id;
        __syncthreads();
        okey = sk[buf][tid ^ j];
        oid = si[buf][tid ^ j];
        buf ^= 1;  // the next exchange writes the other buffer: one barrier is enough
      } else {
        okey = __shfl_xor_sync(0xFFFFFFFFu, key, j);
        oid = __shfl_xor_sync(0xFFFFFFFFu, id, j);
      }
      const bool greater = key > okey || (key == okey && id > oid);
      if ((((tid & j) == 0) == ((tid & k) == 0)) == greater) {
        key = okey;
        id = oid;
      }
    }
  keys[g] = key;
  if (g < n) idx[g] = (int32_t)(blockIdx.x * kChunk + id);
}

// Place of each particle among all chunks: its place in its own plus, of every
// other chunk, the number of smaller keys (of earlier chunks also the equal
// ones).  A block places 32 consecutive keys of one chunk, its warps each
// counting in every kRankWarps-th chunk: the lanes of a warp search the same
// chunk for neighbouring keys, so their probes mostly share a cache line.
__global__ void __launch_bounds__(32 * kRankWarps) k_rank_gather(
    const d4 *__restrict__ posm, int64_t n, const uint64_t *__restrict__ keys,
    const int32_t *__restrict__ idx, int chunks, int32_t *__restrict__ perm,
    d4 *__restrict__ sposm) {
  chain_begin();
  __shared__ int count[kRankWarps][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t g = blockIdx.x * (int64_t)32 + lane;
  const uint64_t key = keys[g];  // the keys are padded to whole chunks
  const int own = (int)(g / kChunk);
  int rank = 0;
#pragma unroll 4
  for (int c = warp; c < chunks; c += kRankWarps) {
    const uint64_t *k = keys + (int64_t)c * kChunk;
    const uint64_t lim = key + (c < own);  // count keys below lim (keys have 63 bits)
    int pos = 0;
#pragma unroll
    for (int h = kChunk / 2; h > 0; h >>= 1)
      if (k[pos + h - 1] < lim) pos += h;
    if (k[pos] < lim) pos++;
    rank += c == own ? (int)(g % kChunk) : pos;
  }
  count[warp][lane] = rank;
  __syncthreads();
  if (warp != 0 || g >= n) return;
#pragma unroll
  for (int w = 1; w < kRankWarps; w++) rank += count[w][lane];
  const int i = idx[g];
  perm[rank] = i;
  sposm[rank] = posm[i];
}

__global__ void __launch_bounds__(kBT) k_gather_posm(const d4 *__restrict__ posm,
                                                     const int32_t *__restrict__ perm, int64_t n,
                                                     d4 *__restrict__ sposm) {
  for (int64_t s = blockIdx.x * (int64_t)kBT + threadIdx.x; s < n; s += (int64_t)gridDim.x * kBT)
    sposm[s] = posm[perm[s]];
}

unsigned grid(int64_t n) {
  int64_t g = (n + kBT - 1) / kBT;
  if (g > 152 * 16) g = 152 * 16;
  return (unsigned)(g < 1 ? 1 : g);
}

// whole chunks
int64_t padded(int64_t n) { return (n + kChunk - 1) / kChunk * kChunk; }
size_t align256(size_t b) { return (b + 255) & ~(size_t)255; }

size_t sort_temp_bytes(int64_t n) {
  size_t bytes = 0;
  cub::DeviceRadixSort::SortPairs(nullptr, bytes, (const uint64_t *)nullptr, (uint64_t *)nullptr,
                                  (const int32_t *)nullptr, (int32_t *)nullptr, (int)n, 0,
                                  3 * kCellBits);
  return bytes;
}

}  // namespace

// Scratch layout: bbox partials | keys in | keys out | identity indices | sort temp.
size_t order_scratch_bytes(int64_t n) {
  return align256(sizeof(uint64_t) * 6 * kBboxBlocks) + 2 * align256(sizeof(uint64_t) * padded(n)) +
         align256(sizeof(int32_t) * n) + align256(sort_temp_bytes(n));
}

cudaError_t launch_spatial_order(const d4 *posm, int64_t n, void *scratch, int32_t *perm,
                                 d4 *sposm, cudaStream_t st) {
  if (n > 0x7fffffff) return cudaErrorInvalidValue;
  char *p = (char *)scratch;
  uint64_t *bb = (uint64_t *)p;
  p += align256(sizeof(uint64_t) * 6 * kBboxBlocks);
  uint64_t *kin = (uint64_t *)p;
  p += align256(sizeof(uint64_t) * padded(n));
  uint64_t *kout = (uint64_t *)p;
  p += align256(sizeof(uint64_t) * padded(n));
  int32_t *idx = (int32_t *)p;
  p += align256(sizeof(int32_t) * n);
  const int nb = (int)std::min<int64_t>(kBboxBlocks, (n + kBT - 1) / kBT);
  cudaError_t e = launch_chained(k_bbox_partial, dim3(nb), kBT, st, posm, n, bb);
  if (e != cudaSuccess) return e;
  if (n <= kRankMax) {
    const int chunks = (int)(padded(n) / kChunk);
    e = launch_chained(k_sort_chunk, dim3(chunks), kChunk, st, posm, n, bb, nb, kin, idx);
    if (e != cudaSuccess) return e;
    return launch_chained(k_rank_gather, dim3((unsigned)((n + 31) / 32)), 32 * kRankWarps, st, posm,
                          n, kin, idx, chunks, perm, sposm);
  }
  k_morton_keys<<<grid(n), kBT, 0, st>>>(posm, n, bb, nb, kin, idx);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  size_t tb = sort_temp_bytes(n);
  e = cub::DeviceRadixSort::SortPairs(p, tb, kin, kout, idx, perm, (int)n, 0, 3 * kCellBits, st);
  if (e != cudaSuccess) return e;
  k_gather_posm<<<grid(n), kBT, 0, st>>>(posm, perm, n, sposm);
  return cudaGetLastError();
}

}  // namespace nb
