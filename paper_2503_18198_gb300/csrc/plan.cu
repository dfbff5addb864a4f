// plan.cu -- building the mode-specific tensor copies and their partitions.
//
// Sec. III-C keeps one COO copy of the tensor per output mode d, ordered for
// that mode; Sec. III-B2 orders the nonzeros by the output-mode index and
// Sec. III-B1 / III-B2 split them into kappa partitions, one per SM.
//
// Ordering used for copy d: (c_d, then c_w for w != d in ascending w, then the
// input position), i.e. a stable sort.  It is built with a device LSD radix
// sort whose digits are slices of one coordinate, at most 10 bits each (a
// 20-bit coordinate: two passes):
//   * copy 0: the full lexicographic key (c_0, c_1, ..., c_{N-1}) packed into
//     64-bit words (several words, least significant first, when the index
//     bits exceed 64), payload = input position; the records are decoded from
//     the sorted keys, only the values are gathered;
//   * copy d >= 1: a stable sort of copy 0 by c_d alone, its keys read from
//     copy 0's records in the first pass.  Among nonzeros with equal c_d, copy
//     0's order is lexicographic on the remaining modes in ascending order,
//     which is exactly the tie-break of copy d.
// Records of copy d hold [c_d, other indices ascending, value bits, padding].
#include <algorithm>
#include <utility>
#include <vector>

#include "plan.cuh"

namespace spm {
namespace {

constexpr int RS_WARPS = 16;
constexpr int RS_THREADS = RS_WARPS * 32;
// Pairs per thread of a tile: 16, or 4 while that leaves few tiles (up to 2^20
// pairs: a tile's chain of ranks is short and there are four times the blocks).
constexpr int RS_ITEMS = 16, RS_ITEMS_SMALL = 4;
constexpr int64_t RS_SMALL = 1 << 20;
inline int rs_tile(int64_t n) { return RS_THREADS * (n <= RS_SMALL ? RS_ITEMS_SMALL : RS_ITEMS); }
// Tiles of n pairs, and the most of any count up to cap.
inline int64_t rs_tiles(int64_t n) { return (n + rs_tile(n) - 1) / rs_tile(n); }
inline int64_t rs_tiles_cap(int64_t cap) {
  const int64_t small = rs_tiles(cap < RS_SMALL ? cap : RS_SMALL);
  return rs_tiles(cap) > small ? rs_tiles(cap) : small;
}
constexpr int RS_BITS = 10;  // widest digit
constexpr int RS_BINS = 1 << RS_BITS;

struct IdxPtrs {
  const int32_t* p[SPM_MAX_MODES];
};

// ---------------------------------------------------------------------------
// LSD radix sort of (key, int32 payload) pairs, up to 10 bits per pass, stable.
// A pass is bound by memory: keys read for the tile histograms, pairs read and
// written by the scatter.  The scatter ranks its tile of 8192 in registers and
// writes it out from shared memory in digit order, so that the 8 or more pairs
// of a digit leave as one run.  50M pairs of 64-bit keys, 10 bits: 630 us a
// pass (8 bits straight from registers: 990 us); 32-bit keys 530 (800).
// ---------------------------------------------------------------------------

template <typename K, int ITEMS>
__global__ void __launch_bounds__(RS_THREADS)
    rs_hist_kernel(const K* __restrict__ keys, int64_t stride, int64_t n, int shift, int width,
                   uint32_t* __restrict__ hist, int ntiles) {
  __shared__ uint32_t cnt[RS_BINS];
  const int bins = 1 << width;
  for (int b = threadIdx.x; b < bins; b += RS_THREADS) cnt[b] = 0;
  __syncthreads();
  const int64_t base = (int64_t)blockIdx.x * (RS_THREADS * ITEMS) + threadIdx.x;
  K key[ITEMS];
#pragma unroll
  for (int i = 0; i < ITEMS; ++i) {
    const int64_t k = base + i * RS_THREADS;
    key[i] = k < n ? keys[k * stride] : K(0);
  }
#pragma unroll
  for (int i = 0; i < ITEMS; ++i)
    if (base + i * RS_THREADS < n) atomicAdd(&cnt[(unsigned)(key[i] >> shift) & (bins - 1)], 1u);
  __syncthreads();
  for (int b = threadIdx.x; b < bins; b += RS_THREADS) hist[(int64_t)b * ntiles + blockIdx.x] = cnt[b];
}

// One block per digit: exclusive scan of hist[d][0..nblocks) in place and the
// digit total into dtot[d].
__global__ void __launch_bounds__(1024)
    rs_scan_rows_kernel(uint32_t* __restrict__ hist, int nblocks, uint32_t* __restrict__ dtot) {
  __shared__ uint32_t wsum[32];
  __shared__ uint32_t carry;
  uint32_t* row = hist + (int64_t)blockIdx.x * nblocks;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nwarps = blockDim.x >> 5;
  if (threadIdx.x == 0) carry = 0;
  __syncthreads();
  for (int base = 0; base < nblocks; base += blockDim.x) {
    const int i = base + threadIdx.x;
    const uint32_t v = i < nblocks ? row[i] : 0u;
    uint32_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      uint32_t y = __shfl_up_sync(SPM_FULL_MASK, x, o);
      if (lane >= o) x += y;
    }
    if (lane == 31) wsum[warp] = x;
    __syncthreads();
    if (warp == 0) {
      uint32_t s = lane < nwarps ? wsum[lane] : 0u;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        uint32_t y = __shfl_up_sync(SPM_FULL_MASK, s, o);
        if (lane >= o) s += y;
      }
      wsum[lane] = s;
    }
    __syncthreads();
    const uint32_t excl = carry + (warp ? wsum[warp - 1] : 0u) + x - v;
    if (i < nblocks) row[i] = excl;
    __syncthreads();
    if (threadIdx.x == blockDim.x - 1) carry = excl + v;
    __syncthreads();
  }
  if (threadIdx.x == 0) dtot[blockIdx.x] = carry;
}

template <typename K, int ITEMS>
struct ScatterSmem {
  K keys[RS_THREADS * ITEMS];                       // the tile in digit order, then its payloads
  unsigned short wcnt[RS_WARPS][RS_BINS];  // per warp and digit: count, then first place in the tile
  uint32_t gbase[RS_BINS];               // global place of a digit's run minus its place in the tile
};

// Exclusive block scan of one value per thread.
__device__ __forceinline__ uint32_t rs_block_exclusive(uint32_t v, uint32_t* wsum) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(SPM_FULL_MASK, x, o);
    if (lane >= o) x += y;
  }
  __syncthreads();
  if (lane == 31) wsum[warp] = x;
  __syncthreads();
  uint32_t pre = 0;
#pragma unroll
  for (int w = 0; w < RS_WARPS; ++w) pre += w < warp ? wsum[w] : 0u;
  return pre + x - v;
}

// One tile: pairs (keys[k * stride], vals ? vals[k] : k) to their places by
// digit.  hist: the tile histograms scanned along the tiles, dtot the digit
// totals (both null: the only tile).  keys_out may be null.
template <typename K, int ITEMS>
__global__ void __launch_bounds__(RS_THREADS, 2)
    rs_scatter_kernel(const K* __restrict__ keys_in, int64_t stride,
                      const int32_t* __restrict__ vals_in, K* __restrict__ keys_out,
                      int32_t* __restrict__ vals_out, int64_t n, int shift, int width,
                      const uint32_t* __restrict__ hist, const uint32_t* __restrict__ dtot,
                      int ntiles) {
  extern __shared__ __align__(16) unsigned char smem_rs[];
  constexpr int TILE = RS_THREADS * ITEMS;
  ScatterSmem<K, ITEMS>& sm = *reinterpret_cast<ScatterSmem<K, ITEMS>*>(smem_rs);
  __shared__ uint32_t wsum[RS_WARPS];
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const unsigned bins = 1u << width;
  for (unsigned x = t; x < RS_WARPS * RS_BINS / 2; x += RS_THREADS)
    reinterpret_cast<uint32_t*>(&sm.wcnt[0][0])[x] = 0;
  __syncthreads();
  const unsigned lt = (1u << lane) - 1u;
  const int64_t tbase = (int64_t)blockIdx.x * TILE;
  const int64_t wbase = tbase + (int64_t)warp * (32 * ITEMS) + lane;
  const int nv = (int)(n - tbase < TILE ? n - tbase : TILE);
  // rank of each pair among its warp's pairs of the same digit so far; places
  // past the end take the last digit and end up past the tile's last pair
  K key[ITEMS];
  uint32_t rk[ITEMS / 2];  // two 16-bit places per word
#pragma unroll
  for (int i = 0; i < ITEMS; ++i) {
    const int64_t k = wbase + i * 32;
    key[i] = k < n ? keys_in[k * stride] : ~K(0);
  }
#pragma unroll
  for (int i = 0; i < ITEMS; ++i) {
    const unsigned d = (unsigned)(key[i] >> shift) & (bins - 1);
    unsigned peers = SPM_FULL_MASK;
#pragma unroll
    for (int b = 0; b < RS_BITS; ++b) {
      const bool bit = (d >> b) & 1u;
      const unsigned with = __ballot_sync(SPM_FULL_MASK, bit);
      peers &= bit ? with : ~with;
    }
    const unsigned r = __popc(peers & lt);
    const unsigned before = sm.wcnt[warp][d];
    __syncwarp();
    if (r == 0) sm.wcnt[warp][d] = (unsigned short)(before + __popc(peers));
    __syncwarp();
    if (i & 1) rk[i / 2] |= (before + r) << 16;
    else rk[i / 2] = before + r;
  }
  __syncthreads();
  // digits 2t and 2t + 1: counts of the warps before, then of the digits before
  unsigned c0 = 0, c1 = 0;
  const unsigned b0 = 2 * t, b1 = 2 * t + 1;
  if (b0 < bins) {
#pragma unroll
    for (int w = 0; w < RS_WARPS; ++w) {
      const uint32_t c = *reinterpret_cast<const uint32_t*>(&sm.wcnt[w][b0]);
      *reinterpret_cast<uint32_t*>(&sm.wcnt[w][b0]) = c0 | (c1 << 16);
      c0 += c & 0xffffu;
      c1 += c >> 16;
    }
  }
  const uint32_t lo = rs_block_exclusive(c0 + c1, wsum);
  uint32_t go = 0, t0 = 0;
  if (hist) {
    t0 = b0 < bins ? dtot[b0] : 0u;
    const uint32_t t1 = b1 < bins ? dtot[b1] : 0u;
    go = rs_block_exclusive(t0 + t1, wsum);
  }
  if (b0 < bins) {
#pragma unroll
    for (int w = 0; w < RS_WARPS; ++w) {
      const uint32_t c = *reinterpret_cast<const uint32_t*>(&sm.wcnt[w][b0]);
      *reinterpret_cast<uint32_t*>(&sm.wcnt[w][b0]) =
          ((c & 0xffffu) + lo) | (((c >> 16) + lo + c0) << 16);
    }
    sm.gbase[b0] = hist ? go + hist[(int64_t)b0 * ntiles + blockIdx.x] - lo : 0u;
    if (b1 < bins)
      sm.gbase[b1] = hist ? go + t0 + hist[(int64_t)b1 * ntiles + blockIdx.x] - (lo + c0) : 0u;
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < ITEMS; ++i) {
    const unsigned d = (unsigned)(key[i] >> shift) & (bins - 1);
    const unsigned pos = sm.wcnt[warp][d] + ((rk[i / 2] >> (16 * (i & 1))) & 0xffffu);
    sm.keys[pos] = key[i];
    rk[i / 2] = (i & 1) ? (rk[i / 2] & 0xffffu) | (pos << 16) : (rk[i / 2] & 0xffff0000u) | pos;
  }
  __syncthreads();
  uint32_t g[ITEMS];
#pragma unroll
  for (int i = 0; i < ITEMS; ++i) {
    const int x = t + i * RS_THREADS;
    if (x < nv) {
      const K k = sm.keys[x];
      g[i] = sm.gbase[(unsigned)(k >> shift) & (bins - 1)] + x;
      if (keys_out) keys_out[g[i]] = k;
    }
  }
  __syncthreads();
  int32_t* sv = reinterpret_cast<int32_t*>(sm.keys);
#pragma unroll
  for (int i = 0; i < ITEMS; ++i) {
    const int64_t k = wbase + i * 32;
    if (k < n) sv[(rk[i / 2] >> (16 * (i & 1))) & 0xffffu] = vals_in ? vals_in[k] : (int32_t)k;
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < ITEMS; ++i) {
    const int x = t + i * RS_THREADS;
    if (x < nv) vals_out[g[i]] = sv[x];
  }
}

struct SortScratch {
  uint32_t* hist = nullptr;
  uint32_t* dtot = nullptr;
};

template <typename K, int ITEMS>
spm_status radix_pass_t(const K* keys, int64_t stride, const int32_t* vals, K* keys_out,
                        int32_t* vals_out, int64_t n, int shift, int width, const SortScratch& sc,
                        cudaStream_t s) {
  const int ntiles = (int)ceil_div<int64_t>(n, RS_THREADS * ITEMS);
  constexpr int smem = (int)sizeof(ScatterSmem<K, ITEMS>);
  SPM_CUDA_TRY(cudaFuncSetAttribute(rs_scatter_kernel<K, ITEMS>,
                                    cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
  if (ntiles > 1) {
    rs_hist_kernel<K, ITEMS><<<ntiles, RS_THREADS, 0, s>>>(keys, stride, n, shift, width, sc.hist,
                                                          ntiles);
    const int st = std::min(1024, (ntiles + 31) / 32 * 32);
    rs_scan_rows_kernel<<<1 << width, st, 0, s>>>(sc.hist, ntiles, sc.dtot);
  }
  rs_scatter_kernel<K, ITEMS><<<ntiles, RS_THREADS, smem, s>>>(
      keys, stride, vals, keys_out, vals_out, n, shift, width, ntiles > 1 ? sc.hist : nullptr,
      ntiles > 1 ? sc.dtot : nullptr, ntiles);
  SPM_CUDA_TRY(cudaGetLastError());
  return SPM_OK;
}

// One stable pass by digit (key >> shift) & (2^width - 1).
template <typename K>
spm_status radix_pass(const K* keys, int64_t stride, const int32_t* vals, K* keys_out,
                      int32_t* vals_out, int64_t n, int shift, int width, const SortScratch& sc,
                      cudaStream_t s) {
  return n <= RS_SMALL ? radix_pass_t<K, RS_ITEMS_SMALL>(keys, stride, vals, keys_out, vals_out, n,
                                                        shift, width, sc, s)
                       : radix_pass_t<K, RS_ITEMS>(keys, stride, vals, keys_out, vals_out, n, shift,
                                                   width, sc, s);
}

// Digits of a field of `bits` bits: count and width of each (the last may reach
// past the field: the bits there are zero or belong to what is sorted later).
inline int digit_count(int bits) { return ceil_div(bits, RS_BITS); }
inline int digit_width(int bits) { return bits > 0 ? ceil_div(bits, digit_count(bits)) : 0; }

// Sorts (keys, vals) by the `bits` bits of the keys from `shift` on, stably.
// The result ends in (keys, vals) (buffers are swapped internally as needed).
// vals_iota: the payloads of the first pass are the positions.
template <typename K>
spm_status radix_sort_pairs(K*& keys, int32_t*& vals, K*& keys_alt, int32_t*& vals_alt,
                            int64_t n, int bits, bool vals_iota, const SortScratch& sc,
                            cudaStream_t s) {
  const int nd = digit_count(bits), w = digit_width(bits);
  for (int p = 0; p < nd; ++p) {
    const int wp = std::min(w, bits - p * w);
    SPM_TRY(radix_pass<K>(keys, 1, vals_iota && p == 0 ? nullptr : vals, keys_alt, vals_alt, n,
                          p * w, wp, sc, s));
    std::swap(keys, keys_alt);
    std::swap(vals, vals_alt);
  }
  return SPM_OK;
}

// ---------------------------------------------------------------------------
// Small element-wise kernels.
// ---------------------------------------------------------------------------

// Every index against its dimension, and (key non-null) the packed key of each
// nonzero: mode w from bit spec.shift[w] on, for w in [spec.lo, spec.hi].
struct PackSpec {
  int lo, hi;
  int shift[SPM_MAX_MODES];
};
struct DimLimits {
  uint32_t d[SPM_MAX_MODES];  // dims, each below 2^31
};
__global__ void validate_pack_kernel(IdxPtrs idx, int nmodes, DimLimits dims, int64_t n,
                                     PackSpec spec, unsigned long long* __restrict__ key,
                                     int* __restrict__ err) {
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n;
       k += (int64_t)gridDim.x * blockDim.x) {
    bool bad = false;
    unsigned long long v = 0;
    for (int w = 0; w < nmodes; ++w) {
      const int32_t c = idx.p[w][k];
      bad |= (uint32_t)c >= dims.d[w];  // negative indices too
      if (w >= spec.lo && w <= spec.hi) v |= (unsigned long long)(uint32_t)c << spec.shift[w];
    }
    if (key) key[k] = v;
    if (bad) atomicOr(err, DEV_ERR_INDEX);
  }
}

// key[k] = packed (c_lo, ..., c_hi) of input position perm[k] (identity if
// perm == nullptr).
__global__ void pack_keys_kernel(IdxPtrs idx, PackSpec spec, const int32_t* __restrict__ perm,
                                 int64_t n, unsigned long long* __restrict__ key) {
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n;
       k += (int64_t)gridDim.x * blockDim.x) {
    const int64_t src = perm ? perm[k] : k;
    unsigned long long v = 0;
    for (int w = spec.lo; w <= spec.hi; ++w)
      v |= (unsigned long long)(uint32_t)idx.p[w][src] << spec.shift[w];
    key[k] = v;
  }
}

// Copy-0 records from the input arrays: [c_0, ..., c_{N-1}, val, 0...].
template <int RI>
__global__ void records_from_input_kernel(IdxPtrs idx, const float* __restrict__ vals,
                                          const int32_t* __restrict__ perm, int nmodes,
                                          int64_t n, int4* __restrict__ rec) {
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n;
       k += (int64_t)gridDim.x * blockDim.x) {
    const int64_t src = perm[k];
    int words[4 * RI];
#pragma unroll
    for (int j = 0; j < 4 * RI; ++j) words[j] = 0;
#pragma unroll
    for (int w = 0; w < SPM_MAX_MODES && w < 4 * RI; ++w)
      if (w < nmodes) words[w] = idx.p[w][src];
    // value bits right after the indices
#pragma unroll
    for (int j = 0; j < 4 * RI; ++j)
      if (j == nmodes) words[j] = __float_as_int(vals[src]);
#pragma unroll
    for (int q = 0; q < RI; ++q)
      rec[k * RI + q] = make_int4(words[4 * q], words[4 * q + 1], words[4 * q + 2], words[4 * q + 3]);
  }
}

// Copy-0 records from the sorted packed keys (all modes in one word) and the
// gathered values, with the block partials of |X|^2: repeated cells are
// adjacent and summed before squaring, by the first of them.
struct UnpackSpec {
  int shift[SPM_MAX_MODES];
  unsigned mask[SPM_MAX_MODES];
};
template <int RI>
__global__ void __launch_bounds__(256)
    records_from_keys_kernel(const unsigned long long* __restrict__ key, UnpackSpec spec,
                             const float* __restrict__ vals, const int32_t* __restrict__ perm,
                             int nmodes, int64_t n, int4* __restrict__ rec,
                             double* __restrict__ part) {
  __shared__ double sh[256];
  double acc = 0.0;
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n;
       k += (int64_t)gridDim.x * blockDim.x) {
    const unsigned long long v = key[k];
    const float x = __ldg(vals + perm[k]);
    int words[4 * RI];
#pragma unroll
    for (int j = 0; j < 4 * RI; ++j) {
      words[j] = 0;
      if (j < SPM_MAX_MODES && j < nmodes)
        words[j] = (int)((unsigned)(v >> spec.shift[j]) & spec.mask[j]);
      else if (j == nmodes)
        words[j] = __float_as_int(x);
    }
#pragma unroll
    for (int q = 0; q < RI; ++q)
      rec[k * RI + q] = make_int4(words[4 * q], words[4 * q + 1], words[4 * q + 2], words[4 * q + 3]);
    if (k > 0 && key[k - 1] == v) continue;
    double cell = (double)x;
    for (int64_t q = k + 1; q < n && key[q] == v; ++q) cell += (double)__ldg(vals + perm[q]);
    acc = fma(cell, cell, acc);
  }
  sh[threadIdx.x] = acc;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) part[blockIdx.x] = sh[0];
}

// Copy-d record k from copy-0 record rel[k]: rotate c_d to the front,
// keep the others in ascending mode order; perm_d[k] = perm_0[rel[k]].
template <int RI>
__global__ void records_from_copy0_kernel(const int4* __restrict__ rec0,
                                          const int32_t* __restrict__ perm0,
                                          const int32_t* __restrict__ rel, int nmodes, int d,
                                          int64_t n, int4* __restrict__ recd,
                                          int32_t* __restrict__ permd) {
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n;
       k += (int64_t)gridDim.x * blockDim.x) {
    const int64_t src = rel[k];
    int in[4 * RI], out[4 * RI];
#pragma unroll
    for (int q = 0; q < RI; ++q) {
      const int4 v = rec0[src * RI + q];
      in[4 * q] = v.x; in[4 * q + 1] = v.y; in[4 * q + 2] = v.z; in[4 * q + 3] = v.w;
    }
#pragma unroll
    for (int j = 0; j < 4 * RI; ++j) out[j] = in[j];
    // words 0..d of copy d are (c_d, c_0, ..., c_{d-1}); words > d unchanged.
    if (d > 0) {
      int cd = 0;
#pragma unroll
      for (int j = 0; j < 4 * RI; ++j)
        if (j == d) cd = in[j];
#pragma unroll
      for (int j = 4 * RI - 1; j >= 1; --j)
        if (j <= d) out[j] = in[j - 1];
      out[0] = cd;
    }
#pragma unroll
    for (int q = 0; q < RI; ++q)
      recd[k * RI + q] = make_int4(out[4 * q], out[4 * q + 1], out[4 * q + 2], out[4 * q + 3]);
    permd[k] = perm0[src];
  }
}

// Gather records and permutation of one copy through rel (in -> out).
template <int RI>
__global__ void reorder_copy_kernel(const int4* __restrict__ rec_in, const int32_t* __restrict__ perm_in,
                                    const int32_t* __restrict__ rel, int64_t n,
                                    int4* __restrict__ rec_out, int32_t* __restrict__ perm_out) {
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n;
       k += (int64_t)gridDim.x * blockDim.x) {
    const int64_t src = rel[k];
#pragma unroll
    for (int q = 0; q < RI; ++q) rec_out[k * RI + q] = rec_in[src * RI + q];
    perm_out[k] = perm_in[src];
  }
}

// Scheme 2 offsets floor(z*nnz/kappa).
__global__ void equal_offsets_kernel(int64_t nnz, int kappa, int64_t* __restrict__ off) {
  for (int z = blockIdx.x * blockDim.x + threadIdx.x; z <= kappa; z += gridDim.x * blockDim.x)
    off[z] = ((int64_t)z * nnz) / kappa;
}

// Row degree from the runs of equal c_d in a copy sorted by c_d.
template <int RI>
__global__ void row_degree_kernel(const int4* __restrict__ rec, int64_t n,
                                  int32_t* __restrict__ deg) {
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n;
       k += (int64_t)gridDim.x * blockDim.x) {
    const int c = rec[k * RI].x;
    const bool start = (k == 0) || rec[(k - 1) * RI].x != c;
    if (start) {
      // run length by galloping then binary search over the sorted rows
      int64_t lo = k, step = 1, hi = k + 1;
      while (hi < n && rec[hi * RI].x == c) {
        lo = hi;
        hi = k + (step <<= 1);
      }
      if (hi > n) hi = n;
      // rec[lo].x == c, and rec[hi].x != c or hi == n
      while (hi - lo > 1) {
        const int64_t mid = lo + (hi - lo) / 2;
        if (rec[mid * RI].x == c) lo = mid; else hi = mid;
      }
      deg[c] = (int32_t)(hi - k);
    }
  }
}

// Key that orders rows by (degree descending, index ascending); empty rows last.
__global__ void row_order_key_kernel(const int32_t* __restrict__ deg, int64_t I,
                                     unsigned long long* __restrict__ key,
                                     int32_t* __restrict__ row) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < I;
       i += (int64_t)gridDim.x * blockDim.x) {
    const uint32_t dg = (uint32_t)deg[i];
    key[i] = dg ? ((unsigned long long)(0xFFFFFFFFu - dg) << 32) | (unsigned long long)i
                : ~0ull;
    row[i] = (int32_t)i;
  }
}

// Cyclic deal: the t-th row in degree order goes to partition t mod kappa.
__global__ void deal_rows_kernel(const int32_t* __restrict__ row_sorted,
                                 const int32_t* __restrict__ deg, int64_t I, int kappa,
                                 int32_t* __restrict__ part) {
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < I;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int32_t r = row_sorted[t];
    part[r] = deg[r] ? (int32_t)(t % kappa) : -1;
  }
}

template <int RI>
__global__ void part_key_kernel(const int4* __restrict__ rec, const int32_t* __restrict__ part,
                                int64_t n, uint32_t* __restrict__ key) {
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n;
       k += (int64_t)gridDim.x * blockDim.x)
    key[k] = (uint32_t)part[rec[k * RI].x];
}

// off[z] = first position whose (sorted) key is >= z.
__global__ void lower_bound_offsets_kernel(const uint32_t* __restrict__ key, int64_t n,
                                           int kappa, int64_t* __restrict__ off) {
  for (int z = blockIdx.x * blockDim.x + threadIdx.x; z <= kappa; z += gridDim.x * blockDim.x) {
    int64_t lo = 0, hi = n;
    while (lo < hi) {
      const int64_t mid = lo + (hi - lo) / 2;
      if (key[mid] < (uint32_t)z) lo = mid + 1; else hi = mid;
    }
    off[z] = lo;
  }
}

// |X|^2 over copy 0 (fully sorted, so repeated coordinates are adjacent and
// are summed before squaring).  Block partials in FP64, fixed order.
template <int RI>
__global__ void __launch_bounds__(256)
    norm_partial_kernel(const int4* __restrict__ rec, int nmodes, int64_t n,
                        double* __restrict__ part) {
  __shared__ double sh[256];
  double acc = 0.0;
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n;
       k += (int64_t)gridDim.x * blockDim.x) {
    const int* w = reinterpret_cast<const int*>(rec + k * RI);
    bool start = (k == 0);
    if (!start) {
      const int* p = reinterpret_cast<const int*>(rec + (k - 1) * RI);
      for (int j = 0; j < nmodes; ++j) start |= (w[j] != p[j]);
    }
    if (!start) continue;
    double cell = (double)__int_as_float(w[nmodes]);
    for (int64_t q = k + 1; q < n; ++q) {
      const int* x = reinterpret_cast<const int*>(rec + q * RI);
      bool same = true;
      for (int j = 0; j < nmodes; ++j) same &= (x[j] == w[j]);
      if (!same) break;
      cell += (double)__int_as_float(x[nmodes]);
    }
    acc += cell * cell;
  }
  sh[threadIdx.x] = acc;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) part[blockIdx.x] = sh[0];
}

// One warp, fixed order.
__global__ void sum_partials_kernel(const double* __restrict__ part, int n, double* __restrict__ out) {
  double s = 0.0;
  for (int i = threadIdx.x; i < n; i += 32) s += part[i];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(SPM_FULL_MASK, s, o);
  if (threadIdx.x == 0) *out = s;
}

// ---- work units -----------------------------------------------------------

// Scheme 1 / Scheme 2: unit w of partition z starts at
// off[z] + floor((off[z+1] - off[z]) * w / units).
__global__ void units_from_partitions_kernel(const int64_t* __restrict__ off, int kappa, int units,
                                             int64_t* __restrict__ woff) {
  const int64_t P = (int64_t)kappa * units;
  for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j <= P;
       j += (int64_t)gridDim.x * blockDim.x) {
    if (j == P) {
      woff[j] = off[kappa];
    } else {
      const int z = (int)(j / units), w = (int)(j % units);
      woff[j] = off[z] + ((off[z + 1] - off[z]) * w) / units;
    }
  }
}

// Row starts per segment of SEG copy positions (one warp each), and the bitmap
// of non-empty output rows (mask non-null).  The row of copy position k is
// rows[k * stride] (a copy's records, or its sorted keys).
constexpr int SEG = 512;
__global__ void __launch_bounds__(256)
    row_heads_kernel(const int* __restrict__ rows, int64_t stride, int64_t n, int64_t nseg,
                     uint32_t* __restrict__ cnt, uint32_t* __restrict__ mask) {
  const int lane = threadIdx.x & 31;
  for (int64_t g = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; g < nseg;
       g += (int64_t)gridDim.x * (blockDim.x >> 5)) {
    const int64_t base = g * SEG;
    int r[SEG / 32];
#pragma unroll
    for (int i = 0; i < SEG / 32; ++i) {
      const int64_t k = base + i * 32 + lane;
      r[i] = k < n ? rows[k * stride] : -1;
    }
    int last = base > 0 ? rows[(base - 1) * stride] : -1;  // the row before the chunk
    uint32_t c = 0;
#pragma unroll
    for (int i = 0; i < SEG / 32; ++i) {
      int prev = __shfl_up_sync(SPM_FULL_MASK, r[i], 1);
      if (lane == 0) prev = last;
      last = __shfl_sync(SPM_FULL_MASK, r[i], 31);
      const bool head = r[i] >= 0 && r[i] != prev;
      c += __popc(__ballot_sync(SPM_FULL_MASK, head));
      if (head && mask) atomicOr(&mask[r[i] >> 5], 1u << (r[i] & 31));
    }
    if (lane == 0) cnt[g] = c;
  }
}

// Exclusive scan of cnt[0 .. n) in place, total to *total (one block, 4096
// entries a round; cnt is 16-byte aligned).
__global__ void __launch_bounds__(1024)
    seg_scan_kernel(uint32_t* __restrict__ cnt, int64_t n, uint32_t* __restrict__ total) {
  __shared__ uint32_t wsum[32];
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  uint32_t carry = 0;
  auto load = [&](int64_t b) -> uint4 {
    if (b + 4 <= n) return *reinterpret_cast<const uint4*>(cnt + b);
    return make_uint4(b < n ? cnt[b] : 0u, b + 1 < n ? cnt[b + 1] : 0u, b + 2 < n ? cnt[b + 2] : 0u, 0u);
  };
  uint4 v = load(4 * t);
  for (int64_t base = 0; base < n; base += 4096) {
    const int64_t b = base + 4 * t;
    const uint4 ahead = load(b + 4096);
    const uint32_t own = v.x + v.y + v.z + v.w;
    uint32_t x = own;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(SPM_FULL_MASK, x, o);
      if (lane >= o) x += y;
    }
    if (lane == 31) wsum[warp] = x;
    __syncthreads();
    uint32_t y = wsum[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t z = __shfl_up_sync(SPM_FULL_MASK, y, o);
      if (lane >= o) y += z;
    }
    const uint32_t all = __shfl_sync(SPM_FULL_MASK, y, 31);
    const uint32_t pre = __shfl_sync(SPM_FULL_MASK, y, warp > 0 ? warp - 1 : 0);
    const uint32_t e0 = carry + (warp > 0 ? pre : 0u) + x - own;
    const uint4 o = make_uint4(e0, e0 + v.x, e0 + v.x + v.y, e0 + v.x + v.y + v.z);
    if (b + 4 <= n) {
      *reinterpret_cast<uint4*>(cnt + b) = o;
    } else {
      if (b < n) cnt[b] = o.x;
      if (b + 1 < n) cnt[b + 1] = o.y;
      if (b + 2 < n) cnt[b + 2] = o.z;
    }
    carry += all;
    v = ahead;
    __syncthreads();
  }
  if (t == 0) *total = carry;
}

// woff[j] = min{k in [0, n] : C(k) * P >= j * C(n)},
// C(k) = k + row_cost * (row starts before k), C(n) = n + row_cost * heads;
// off[z] = woff[z * units].  One warp per unit: a binary search over the
// segments, then the row starts inside one.  For copies of many nonzeros per
// unit (50M: 78 us); see units_by_position_kernel.
__global__ void __launch_bounds__(256)
    balanced_units_kernel(const int* __restrict__ rows, int64_t stride, int64_t n,
                          const uint32_t* __restrict__ seg, int64_t nseg,
                          const uint32_t* __restrict__ heads, int64_t P, int units, int row_cost,
                          int64_t* __restrict__ woff, int64_t* __restrict__ off) {
  const int lane = threadIdx.x & 31;
  const int64_t Ct = n + (int64_t)row_cost * (int64_t)(*heads);
  for (int64_t j = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; j <= P;
       j += (int64_t)gridDim.x * (blockDim.x >> 5)) {
    const int64_t target = j * Ct;  // compare C(k) * P >= target
    // last segment that starts below the target (none: position 0)
    int64_t lo = -1, hi = nseg;
    while (hi - lo > 1) {
      const int64_t mid = lo + (hi - lo) / 2;
      const int64_t C = mid * SEG + (int64_t)row_cost * (int64_t)seg[mid];
      if (C * P < target) lo = mid; else hi = mid;
    }
    int64_t res = 0;
    if (lo >= 0) {
      const int64_t base = lo * SEG;
      res = base + SEG < n ? base + SEG : n;
      int64_t before = seg[lo];
      int r[SEG / 32];
#pragma unroll
      for (int i = 0; i < SEG / 32; ++i) {
        const int64_t k = base + i * 32 + lane;
        r[i] = k < n ? rows[k * stride] : -1;
      }
      int last = base > 0 ? rows[(base - 1) * stride] : -1;
#pragma unroll
      for (int i = 0; i < SEG / 32; ++i) {
        const int64_t k = base + i * 32 + lane;
        int prev = __shfl_up_sync(SPM_FULL_MASK, r[i], 1);
        if (lane == 0) prev = last;
        last = __shfl_sync(SPM_FULL_MASK, r[i], 31);
        const unsigned hb = __ballot_sync(SPM_FULL_MASK, r[i] >= 0 && r[i] != prev);
        const int64_t C = k + (int64_t)row_cost * (before + __popc(hb & ((1u << lane) - 1u)));
        const unsigned ok = __ballot_sync(SPM_FULL_MASK, k <= n && C * P >= target);
        if (ok) {
          res = base + i * 32 + (__ffs(ok) - 1);
          break;
        }
        before += __popc(hb);
      }
    }
    if (lane == 0) {
      woff[j] = res;
      if (j % units == 0) off[j / units] = res;
    }
  }
}

// The same from the side of the positions, for few nonzeros per unit: position
// k is the first with C(k) * P >= j * C(n) for the units
// floor(C(k - 1) P / C(n)) < j <= floor(C(k) P / C(n)).  One warp per 32
// positions, which counts the row starts before them in its segment (30,000
// nonzeros, 38,912 units: 51 us by search, 47 us with a warp per segment and
// its 16 chains of 64-bit divisions, 6 us so).
__global__ void __launch_bounds__(256)
    units_by_position_kernel(const int* __restrict__ rows, int64_t stride, int64_t n,
                             const uint32_t* __restrict__ seg, int64_t nseg,
                             const uint32_t* __restrict__ heads, int64_t P, int units, int row_cost,
                             int64_t* __restrict__ woff, int64_t* __restrict__ off) {
  const int lane = threadIdx.x & 31;
  const int64_t Ct = n + (int64_t)row_cost * (int64_t)(*heads);
  // positions 0 .. n: position n closes the copy
  for (int64_t q = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; q * 32 <= n;
       q += (int64_t)gridDim.x * (blockDim.x >> 5)) {
    const int64_t g = q / (SEG / 32), base = g * SEG;
    const int chunk = (int)(q % (SEG / 32));
    int r[SEG / 32];
#pragma unroll
    for (int i = 0; i < SEG / 32; ++i) {
      const int64_t k = base + i * 32 + lane;
      r[i] = i <= chunk && k < n ? rows[k * stride] : -1;
    }
    int last = base > 0 ? rows[(base - 1) * stride] : -1;
    int64_t before = g < nseg ? seg[g] : *heads;
    bool prev_head = false;  // whether position 32 q - 1 starts a row
    if (chunk == 0 && base > 0) prev_head = base == 1 || rows[(base - 2) * stride] != last;
    unsigned hb = 0;
#pragma unroll
    for (int i = 0; i < SEG / 32; ++i) {
      if (i <= chunk) {
        int prev = __shfl_up_sync(SPM_FULL_MASK, r[i], 1);
        if (lane == 0) prev = last;
        last = __shfl_sync(SPM_FULL_MASK, r[i], 31);
        hb = __ballot_sync(SPM_FULL_MASK, r[i] >= 0 && r[i] != prev);
        if (i < chunk) {
          before += __popc(hb);
          prev_head = hb >> 31;
        }
      }
    }
    const int64_t k = q * 32 + lane;
    const int64_t C = k + (int64_t)row_cost * (before + __popc(hb & ((1u << lane) - 1u)));
    const int j1 = k <= n ? (int)(C * P / Ct) : (int)P;
    int j0 = __shfl_up_sync(SPM_FULL_MASK, j1, 1);
    if (lane == 0)
      j0 = q == 0 ? -1
                  : (int)((k - 1 + (int64_t)row_cost * (before - (prev_head ? 1 : 0))) * P / Ct);
    const int cnt = k <= n ? j1 - j0 : 0;
    if (cnt > 0 && cnt <= 4) {
      for (int j = j0 + 1; j <= j1; ++j) {
        woff[j] = k;
        if (j % units == 0) off[j / units] = k;
      }
    }
    unsigned many = __ballot_sync(SPM_FULL_MASK, cnt > 4);
    while (many) {
      const int l = __ffs(many) - 1;
      many &= many - 1;
      const int a = __shfl_sync(SPM_FULL_MASK, j0, l), e = __shfl_sync(SPM_FULL_MASK, j1, l);
      for (int j = a + 1 + lane; j <= e; j += 32) {
        woff[j] = q * 32 + l;
        if (j % units == 0) off[j / units] = q * 32 + l;
      }
    }
  }
}

// Bitmap of non-empty output rows of a copy (rows[k * stride] is the row of
// copy position k; every nonzero sets its row's bit).
__global__ void row_mask_kernel(const int* __restrict__ rows, int64_t stride, int64_t n,
                                uint32_t* __restrict__ mask) {
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n;
       k += (int64_t)gridDim.x * blockDim.x) {
    const int r = rows[k * stride];
    if (k == 0 || rows[(k - 1) * stride] != r) atomicOr(&mask[r >> 5], 1u << (r & 31));
  }
}

// Lean copy d: row of each copy position, gathered from copy 0 (word d of
// the copy-0 record is c_d).
__global__ void gather_rows_kernel(const int* __restrict__ rec0, int64_t words, const int32_t* __restrict__ src,
                                   int d, int64_t n, int* __restrict__ rows) {
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n;
       k += (int64_t)gridDim.x * blockDim.x)
    rows[k] = rec0[(int64_t)src[k] * words + d];
}

__global__ void popc_kernel(const uint32_t* __restrict__ mask, int64_t words,
                            unsigned* __restrict__ count) {
  unsigned c = 0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < words;
       i += (int64_t)gridDim.x * blockDim.x)
    c += __popc(mask[i]);
  for (int o = 16; o > 0; o >>= 1) c += __shfl_down_sync(SPM_FULL_MASK, c, o);
  if ((threadIdx.x & 31) == 0 && c) atomicAdd(count, c);
}

int resolved_scheme(int policy, int64_t dim, int kappa) {
  if (policy == (int)(SPM_POLICY_SCHEME2 >> 4)) return 2;
  if (policy == (int)(SPM_POLICY_SCHEME1 >> 4)) return 1;
  if (policy == (int)(SPM_POLICY_ADAPTIVE >> 4)) return dim >= kappa ? 1 : 2;
  return 0;
}

int grid_for(int64_t n, int threads) {
  const int64_t b = ceil_div<int64_t>(n > 0 ? n : 1, threads);
  return (int)std::min<int64_t>(b, 152 * 32);
}

int bits_for(int64_t dim) {
  int b = 0;
  while (b < 63 && ((int64_t)1 << b) < dim) ++b;
  return b;  // enough bits for values 0..dim-1
}

constexpr int NORM_BLOCKS = 1024;

// The rows of copy d in copy order as (pointer, stride): the copy's records,
// or for a lean copy a key array gathered into `scratch` (>= nnz ints).
const int* copy_rows(spmttkrp_plan_s* p, int d, int* scratch, int64_t* stride, cudaStream_t s) {
  const int RI = record_int4s(p->N);
  if (!p->lean || d == 0) {
    *stride = 4 * RI;
    return reinterpret_cast<const int*>(p->mode[d].rec);
  }
  const int64_t n = p->nnz;
  gather_rows_kernel<<<grid_for(n, 256), 256, 0, s>>>(reinterpret_cast<const int*>(p->mode[0].rec),
                                                     4 * RI, p->mode[d].src, d, n, scratch);
  *stride = 1;
  return scratch;
}

// P2 for a copy under the cost-balanced policy (scheme 0) or Scheme 2, and
// for an empty tensor under any policy: partition offsets off[0..kappa] and
// work-unit offsets woff[0..kappa*nu].  rows/stride: the copy's rows in copy
// order.  Scheme 0 leaves the number of distinct rows in *heads and, with
// `mask`, sets the (cleared) bitmap of non-empty rows.  Scratch: seg >=
// ceil(nnz/SEG) words.
void partition_copy(spmttkrp_plan_s* p, int d, const int* rows, int64_t stride, uint32_t* seg,
                    uint32_t* heads, uint32_t* mask, cudaStream_t s) {
  const int T = 256;
  const int64_t n = p->nnz;
  const int units = p->nu;
  const int64_t P = (int64_t)p->kappa * units;
  spm_mode_copy& c = p->mode[d];
  if (c.scheme == 0 && n > 0) {
    // cost-balanced work units over the copy order
    const int64_t nseg = ceil_div<int64_t>(n, SEG);
    row_heads_kernel<<<grid_for(nseg * 32, T), T, 0, s>>>(rows, stride, n, nseg, seg, mask);
    seg_scan_kernel<<<1, 1024, 0, s>>>(seg, nseg, heads);
    if (n < 16 * P)
      units_by_position_kernel<<<grid_for(n + 32, T), T, 0, s>>>(
          rows, stride, n, seg, nseg, heads, P, units, SPM_ROW_COST, c.woff, c.off);
    else
      balanced_units_kernel<<<grid_for((P + 1) * 32, T), T, 0, s>>>(
          rows, stride, n, seg, nseg, heads, P, units, SPM_ROW_COST, c.woff, c.off);
    return;
  }
  equal_offsets_kernel<<<grid_for(p->kappa + 1, T), T, 0, s>>>(n, p->kappa, c.off);
  units_from_partitions_kernel<<<grid_for(P + 1, T), T, 0, s>>>(c.off, p->kappa, units, c.woff);
}

// Entries of the build's sort scratch: the nonzeros, or the rows of the
// longest mode when some mode is partitioned by Scheme 1 (its rows are
// sorted by degree); policy is SPM_POLICY_* >> 4.
int64_t sort_capacity(int N, const int64_t* dims, int64_t nn, int policy, int kappa) {
  int64_t rows = 0;
  for (int w = 0; w < N; ++w) {
    const bool scheme1 = policy == (int)(SPM_POLICY_SCHEME1 >> 4) ||
                         (policy == (int)(SPM_POLICY_ADAPTIVE >> 4) && dims[w] >= kappa);
    if (scheme1) rows = std::max(rows, dims[w]);
  }
  return std::max(nn, rows);
}

// Transient device memory of a build: one allocation.
struct BuildScratch {
  void* base = nullptr;
  unsigned long long *ka = nullptr, *kb = nullptr;  // keys
  int32_t *va = nullptr, *vb = nullptr;             // payloads
  SortScratch sort;
  unsigned* count = nullptr;  // non-empty rows per mode
  // Bytes for `cap` keys; the pieces are laid out when `p` is non-null.
  static size_t layout(int64_t cap, unsigned char* p, BuildScratch* b) {
    size_t at = 0;
    auto take = [&](size_t bytes) {
      unsigned char* q = p ? p + at : nullptr;
      at += (bytes + 255) & ~(size_t)255;
      return q;
    };
    unsigned char* q[7];
    q[0] = take(sizeof(unsigned long long) * (size_t)cap);
    q[1] = take(sizeof(unsigned long long) * (size_t)cap);
    q[2] = take(sizeof(int32_t) * (size_t)cap);
    q[3] = take(sizeof(int32_t) * (size_t)cap);
    q[4] = take(sizeof(uint32_t) * RS_BINS * (size_t)rs_tiles_cap(cap));
    q[5] = take(sizeof(uint32_t) * RS_BINS);
    q[6] = take(sizeof(unsigned) * SPM_MAX_MODES);
    if (b) {
      b->base = p;
      b->ka = reinterpret_cast<unsigned long long*>(q[0]);
      b->kb = reinterpret_cast<unsigned long long*>(q[1]);
      b->va = reinterpret_cast<int32_t*>(q[2]);
      b->vb = reinterpret_cast<int32_t*>(q[3]);
      b->sort.hist = reinterpret_cast<uint32_t*>(q[4]);
      b->sort.dtot = reinterpret_cast<uint32_t*>(q[5]);
      b->count = reinterpret_cast<unsigned*>(q[6]);
    }
    return at;
  }
  cudaStream_t stream = nullptr;
  size_t bytes = 0;
  spm_status alloc(int64_t cap, cudaStream_t s) {
    void* p = nullptr;
    stream = s;
    bytes = layout(cap, nullptr, nullptr);
    SPM_TRY(dev_alloc(&p, bytes));
    layout(cap, static_cast<unsigned char*>(p), this);
    return SPM_OK;
  }
  BuildScratch() = default;
  BuildScratch(const BuildScratch&) = delete;
  BuildScratch& operator=(const BuildScratch&) = delete;
  ~BuildScratch() { release(); }
  // A synchronisation of the stream after it gives large scratch back.
  void release() {
    scratch_free(base, bytes, stream);
    base = nullptr;
  }
};

template <int RI>
spm_status build_copies_t(spmttkrp_plan_s* p, const int32_t* const* idx_in, const float* vals,
                          cudaStream_t s) {
  const int N = p->N;
  const int64_t n = p->nnz;
  IdxPtrs idx{};
  for (int w = 0; w < N; ++w) idx.p[w] = idx_in[w];
  const int T = 256;
  const int G = grid_for(n, T);

  const int64_t nn = n > 0 ? n : 1;
  // the keys, payloads and histograms hold nnz entries, or I_d entries where
  // Scheme 1 sorts the rows of a mode by degree
  const int64_t cap = sort_capacity(N, p->dims, nn, p->policy, p->kappa);
  BuildScratch b;
  SPM_TRY(b.alloc(cap, s));
  const SortScratch& sc = b.sort;

  // modes grouped into <=64-bit key words from the last mode backwards
  int bits[SPM_MAX_MODES];
  for (int w = 0; w < N; ++w) bits[w] = bits_for(p->dims[w]);
  struct Group { int lo, hi; };
  std::vector<Group> groups;
  {
    int hi = N - 1, acc = 0;
    for (int w = N - 1; w >= 0; --w) {
      if (acc + bits[w] > 64) {
        groups.push_back({w + 1, hi});
        hi = w;
        acc = 0;
      }
      acc += bits[w];
    }
    groups.push_back({0, hi});
  }
  auto spec_of = [&](const Group& g) {
    PackSpec spec{};
    spec.lo = g.lo;
    spec.hi = g.hi;
    int sh = 0;
    for (int w = g.hi; w >= g.lo; --w) {
      spec.shift[w] = sh;
      sh += bits[w];
    }
    return spec;
  };

  // Validation: every index within its dimension; and the keys of the first sort.
  if (n > 0) {
    DimLimits lim{};
    for (int w = 0; w < N; ++w) lim.d[w] = (uint32_t)p->dims[w];
    validate_pack_kernel<<<G, T, 0, s>>>(idx, N, lim, n, spec_of(groups[0]), b.ka, p->dev_err);
  }
  int herr = 0;
  SPM_CUDA_TRY(cudaMemcpyAsync(&herr, p->dev_err, sizeof(int), cudaMemcpyDeviceToHost, s));
  SPM_CUDA_TRY(cudaStreamSynchronize(s));
  spm_status st = SPM_OK;
  if (herr & DEV_ERR_INDEX) st = SPM_ERR_INDEX_OUT_OF_RANGE;

  // Allocate the copies (a lean copy: positions into copy 0, padded by 16
  // bytes so that 16-byte-aligned bulk copies of any range stay inside).
  for (int d = 0; d < N && st == SPM_OK; ++d) {
    if (p->lean && d > 0) {
      st = plan_alloc(p, (void**)&p->mode[d].src, sizeof(int32_t) * (size_t)nn + 16);
    } else {
      st = plan_alloc(p, (void**)&p->mode[d].rec, sizeof(int4) * RI * (size_t)nn + 256);
      if (st == SPM_OK) st = plan_alloc(p, (void**)&p->mode[d].perm, sizeof(int32_t) * (size_t)nn);
    }
    if (st == SPM_OK)
      st = plan_alloc(p, (void**)&p->mode[d].off, sizeof(int64_t) * (size_t)(p->kappa + 1));
    if (st == SPM_OK)
      st = plan_alloc(p, (void**)&p->mode[d].woff,
                      sizeof(int64_t) * ((size_t)p->kappa * p->nu + 1));
    if (st == SPM_OK)
      st = plan_alloc(p, (void**)&p->mode[d].rowmask,
                      sizeof(uint32_t) * (size_t)((p->dims[d] + 31) / 32));
  }

  for (int d = 0; d < N; ++d) p->mode[d].scheme = resolved_scheme(p->policy, p->dims[d], p->kappa);
  plan_shapes(p);
  const int units = p->nu;
  const int64_t P = (int64_t)p->kappa * units;
  if (st == SPM_OK) {
    SPM_CUDA_TRY(cudaMemsetAsync(b.count, 0, sizeof(unsigned) * SPM_MAX_MODES, s));
    for (int d = 0; d < N; ++d)
      SPM_CUDA_TRY(cudaMemsetAsync(p->mode[d].rowmask, 0,
                                   sizeof(uint32_t) * (size_t)((p->dims[d] + 31) / 32), s));
  }

  if (st == SPM_OK && n > 0) {
    // ---- copy 0: full lexicographic order, least significant key word first.
    spm_mode_copy& c0 = p->mode[0];
    unsigned long long *ka = b.ka, *kb = b.kb;
    const int32_t* pa = nullptr;  // null: input positions in order
    int32_t* free_perm[2] = {b.va, b.vb};
    for (size_t q = 0; q < groups.size() && st == SPM_OK; ++q) {  // least significant group first
      const Group& g = groups[q];
      const PackSpec spec = spec_of(g);
      if (q > 0) pack_keys_kernel<<<G, T, 0, s>>>(idx, spec, pa, n, ka);
      std::vector<std::pair<int, int>> passes;  // (shift, width)
      for (int w = g.hi; w >= g.lo; --w) {
        const int wd = digit_width(bits[w]);
        for (int x = 0; x < bits[w]; x += wd)
          passes.push_back({spec.shift[w] + x, std::min(wd, bits[w] - x)});
      }
      if (passes.empty() && q + 1 == groups.size()) passes.push_back({0, 1});  // writes the order
      for (size_t x = 0; x < passes.size() && st == SPM_OK; ++x) {
        const bool last = q + 1 == groups.size() && x + 1 == passes.size();
        int32_t* out = last ? c0.perm : free_perm[0];
        st = radix_pass<unsigned long long>(ka, 1, pa, kb, out, n, passes[x].first,
                                            passes[x].second, sc, s);
        std::swap(ka, kb);
        std::swap(free_perm[0], free_perm[1]);
        pa = out;
      }
    }
    if (st == SPM_OK) {
      if (groups.size() == 1) {
        UnpackSpec u{};
        const PackSpec spec = spec_of(groups[0]);
        for (int w = 0; w < N; ++w) {
          u.shift[w] = bits[w] ? spec.shift[w] : 0;
          u.mask[w] = bits[w] ? (unsigned)((1ull << bits[w]) - 1) : 0u;
        }
        records_from_keys_kernel<RI><<<NORM_BLOCKS, 256, 0, s>>>(ka, u, vals, c0.perm, N, n, c0.rec,
                                                               p->norm_part);
      } else {
        records_from_input_kernel<RI><<<G, T, 0, s>>>(idx, vals, c0.perm, N, n, c0.rec);
        // |X|^2 (duplicates summed) from copy 0
        norm_partial_kernel<RI><<<NORM_BLOCKS, 256, 0, s>>>(c0.rec, N, n, p->norm_part);
      }
      sum_partials_kernel<<<1, 32, 0, s>>>(p->norm_part, NORM_BLOCKS, p->normX2);
    }
  } else if (st == SPM_OK) {
    SPM_CUDA_TRY(cudaMemsetAsync(p->normX2, 0, sizeof(double), s));
  }

  // ---- copies d >= 1 (stable sort of copy 0 by c_d), then each copy's
  // partitions (Sec. III-B), work units and bitmap of non-empty rows; copy 0
  // last, because Scheme 1 reorders it
  for (int x = 1; x <= N && st == SPM_OK; ++x) {
    const int d = x % N;
    spm_mode_copy& c = p->mode[d];
    const int* rows = n > 0 ? reinterpret_cast<const int*>(p->mode[0].rec) : nullptr;
    int64_t stride = 4 * RI;
    if (d > 0 && n > 0) {
      uint32_t *ko = reinterpret_cast<uint32_t*>(b.kb), *kf = reinterpret_cast<uint32_t*>(b.ka);
      const uint32_t* ki = reinterpret_cast<const uint32_t*>(rows) + d;
      const int32_t* ri = nullptr;
      int32_t *ro = b.va, *rf = b.vb;
      const int nb = std::max(1, bits[d]), wd = digit_width(nb);
      for (int bit = 0; bit < nb && st == SPM_OK; bit += wd) {
        int32_t* out = p->lean && bit + wd >= nb ? c.src : ro;
        st = radix_pass<uint32_t>(ki, bit == 0 ? stride : 1, ri, ko, out, n, bit,
                                  std::min(wd, nb - bit), sc, s);
        ki = ko;
        ri = out;
        std::swap(ko, kf);
        std::swap(ro, rf);
      }
      if (st != SPM_OK) break;
      if (!p->lean)
        records_from_copy0_kernel<RI><<<G, T, 0, s>>>(p->mode[0].rec, p->mode[0].perm, ri, N, d, n,
                                                       c.rec, c.perm);
      rows = reinterpret_cast<const int*>(ki);
      stride = 1;
    }
    if (c.scheme != 1 || n == 0) {
      partition_copy(p, d, rows, stride, sc.hist, b.count + d, c.rowmask, s);
      if (c.scheme != 0 && n > 0) {
        row_mask_kernel<<<G, T, 0, s>>>(rows, stride, n, c.rowmask);
        const int64_t words = (p->dims[d] + 31) / 32;
        popc_kernel<<<grid_for(words, T), T, 0, s>>>(c.rowmask, words, b.count + d);
      }
      continue;
    }
    // Scheme 1: degree-ordered cyclic deal of the rows, copy ordered by partition.
    const int64_t I = p->dims[d];
    int32_t* deg = nullptr;
    int32_t* part = nullptr;
    int4* rec_tmp = nullptr;
    int32_t* perm_tmp = nullptr;
    SPM_CUDA_TRY(cudaMallocAsync((void**)&deg, sizeof(int32_t) * I, s));
    SPM_CUDA_TRY(cudaMallocAsync((void**)&part, sizeof(int32_t) * I, s));
    SPM_CUDA_TRY(cudaMallocAsync((void**)&rec_tmp, sizeof(int4) * RI * (size_t)n, s));
    SPM_CUDA_TRY(cudaMallocAsync((void**)&perm_tmp, sizeof(int32_t) * (size_t)n, s));
    SPM_CUDA_TRY(cudaMemsetAsync(deg, 0, sizeof(int32_t) * I, s));
    row_degree_kernel<RI><<<G, T, 0, s>>>(c.rec, n, deg);
    {
      unsigned long long *ka = b.ka, *kb = b.kb;
      int32_t *ra = b.va, *rb = b.vb;
      row_order_key_kernel<<<grid_for(I, T), T, 0, s>>>(deg, I, ka, ra);
      st = radix_sort_pairs<unsigned long long>(ka, ra, kb, rb, I, 64, false, sc, s);
      if (st == SPM_OK) deal_rows_kernel<<<grid_for(I, T), T, 0, s>>>(ra, deg, I, p->kappa, part);
    }
    if (st == SPM_OK) {
      uint32_t* ka32 = reinterpret_cast<uint32_t*>(b.ka);
      uint32_t* kb32 = reinterpret_cast<uint32_t*>(b.kb);
      int32_t *ra = b.va, *rb = b.vb;
      part_key_kernel<RI><<<G, T, 0, s>>>(c.rec, part, n, ka32);
      st = radix_sort_pairs<uint32_t>(ka32, ra, kb32, rb, n, std::max(1, bits_for(p->kappa)), true,
                                      sc, s);
      if (st == SPM_OK) {
        reorder_copy_kernel<RI><<<G, T, 0, s>>>(c.rec, c.perm, ra, n, rec_tmp, perm_tmp);
        SPM_CUDA_TRY(cudaMemcpyAsync(c.rec, rec_tmp, sizeof(int4) * RI * (size_t)n,
                                     cudaMemcpyDeviceToDevice, s));
        SPM_CUDA_TRY(cudaMemcpyAsync(c.perm, perm_tmp, sizeof(int32_t) * (size_t)n,
                                     cudaMemcpyDeviceToDevice, s));
        lower_bound_offsets_kernel<<<grid_for(p->kappa + 1, T), T, 0, s>>>(ka32, n, p->kappa,
                                                                          c.off);
        units_from_partitions_kernel<<<grid_for(P + 1, T), T, 0, s>>>(c.off, p->kappa, units,
                                                                      c.woff);
        row_mask_kernel<<<G, T, 0, s>>>(reinterpret_cast<const int*>(c.rec), 4 * RI, n, c.rowmask);
        const int64_t words = (I + 31) / 32;
        popc_kernel<<<grid_for(words, T), T, 0, s>>>(c.rowmask, words, b.count + d);
      }
    }
    SPM_CUDA_TRY(cudaFreeAsync(deg, s));
    SPM_CUDA_TRY(cudaFreeAsync(part, s));
    SPM_CUDA_TRY(cudaFreeAsync(rec_tmp, s));
    SPM_CUDA_TRY(cudaFreeAsync(perm_tmp, s));
  }
  unsigned h_cnt[SPM_MAX_MODES] = {};
  if (st == SPM_OK)
    SPM_CUDA_TRY(cudaMemcpyAsync(h_cnt, b.count, sizeof(unsigned) * SPM_MAX_MODES,
                                 cudaMemcpyDeviceToHost, s));
  SPM_CUDA_TRY(cudaGetLastError());
  b.release();
  SPM_CUDA_TRY(cudaStreamSynchronize(s));
  for (int d = 0; d < N; ++d) p->mode[d].empty_rows = p->dims[d] - (int64_t)h_cnt[d];
  return st;
}

}  // namespace

void plan_shapes(spmttkrp_plan_s* p) {
  const int sms = sm_count();
  for (int d = 0; d < p->N; ++d) {
    spm_mode_copy& c = p->mode[d];
    const MttkrpShape x = mttkrp_shape(c.scheme, p->nnz, p->kappa, p->nu, sms);
    c.kx = x.kx;
    c.nx = x.nx;
  }
}

void plan_bytes_estimate(int N, const int64_t* dims, int64_t nnz, int R, int kappa, bool als,
                         bool lean, size_t* resident, size_t* transient, bool fibre, int policy,
                         bool bf16) {
  // mirrors the plan_alloc calls of spmttkrp_plan, build_copies and
  // ensure_als_state (each allocation of 0 bytes counts 16)
  const int RI = record_int4s(N);
  const int nu = fibre ? 32 * fibre_slots(R) : SPM_UNITS_PER_PARTITION(R);
  const int64_t nn = nnz > 0 ? nnz : 1;
  int64_t Imax = 1;
  for (int w = 0; w < N; ++w) Imax = std::max(Imax, dims[w]);
  const size_t nb = (size_t)boundary_blocks(nnz, kappa, sm_count());
  size_t b = 2 * sizeof(int) + sizeof(double);  // dev_err, normX2
  b += sizeof(float) * 2 * nb * R + sizeof(int) * 4 * nb;
  b += sizeof(double) * NORM_BLOCKS;
  for (int d = 0; d < N; ++d) {
    if (lean && d > 0) {
      b += sizeof(int32_t) * (size_t)nn + 16;
    } else if (fibre) {
      // at most one fibre per nonzero: an upper bound (the count is data-dependent)
      b += sizeof(int2) * (size_t)(2 * (size_t)(nnz > 0 ? nnz : 0) + 2);
      b += sizeof(FibreUnit) * (size_t)kappa * nu;
      b += sizeof(int32_t) * (size_t)nn;
    } else {
      b += sizeof(int4) * RI * (size_t)nn + 256;
      b += sizeof(int32_t) * (size_t)nn;
    }
    b += sizeof(int64_t) * (size_t)(kappa + 1);
    b += sizeof(int64_t) * ((size_t)kappa * nu + 1);
    b += sizeof(uint32_t) * (size_t)((dims[d] + 31) / 32);
  }
  if (als) {
    const size_t gb = (size_t)std::max(1, sm_count()) * 4;
    const size_t RR = (size_t)R * R;
    b += sizeof(double) * RR * N + sizeof(double) * RR * gb;
    b += sizeof(float) * 2 * RR + sizeof(double) * R * gb * 2 + sizeof(double) * 2 * R;
    b += sizeof(float) * R * gb + als_wdig_bytes(R);  // column maxima of Z, W digit tiles
    b += sizeof(float) * (size_t)Imax * R * 2;
    if (als_splits(bf16, fibre, nnz, kappa, nu, sm_count()))
      b += (sizeof(float) * R + sizeof(int)) * 2 * (size_t)kappa * nu + sizeof(int) * (size_t)kappa;
  }
  *resident = b;
  // stream-ordered scratch of the build (keys, payloads, histograms)
  const int64_t cap = sort_capacity(N, dims, nn, policy, kappa);
  *transient = BuildScratch::layout(cap, nullptr, nullptr);
  if (fibre)  // the record copies live until every fibre stream is built
    *transient = std::max<size_t>(*transient, (sizeof(int4) * RI + 256) * (size_t)nn * N +
                                                  sizeof(int32_t) * (size_t)nn);
}

spm_status plan_repartition(spmttkrp_plan_s* p, int kappa, cudaStream_t s) {
  if (kappa < 1 || kappa > 0xFFFF) return SPM_ERR_INVALID_ARG;
  if (p->fibre) return SPM_ERR_UNSUPPORTED;  // work units are baked into the fibre streams
  if (p->policy != (int)(SPM_POLICY_BALANCED >> 4) && p->policy != (int)(SPM_POLICY_SCHEME2 >> 4))
    return SPM_ERR_UNSUPPORTED;
  if (kappa == p->kappa) return SPM_OK;
  if (kappa > p->kappa_cap) {
    // the old arrays may still be read by queued work
    SPM_CUDA_TRY(cudaStreamSynchronize(s));
    for (int d = 0; d < p->N; ++d) {
      SPM_TRY(plan_realloc(p, (void**)&p->mode[d].off, sizeof(int64_t) * (size_t)(kappa + 1)));
      SPM_TRY(plan_realloc(p, (void**)&p->mode[d].woff,
                           sizeof(int64_t) * ((size_t)kappa * p->nu + 1)));
    }
    const size_t nb = (size_t)boundary_blocks(p->nnz, kappa, sm_count());
    SPM_TRY(plan_realloc(p, (void**)&p->cta_part, sizeof(float) * 2 * nb * p->R));
    SPM_TRY(plan_realloc(p, (void**)&p->cta_meta, sizeof(int) * 4 * nb));
    p->kappa_cap = kappa;
  }
  p->kappa = kappa;
  plan_shapes(p);
  const int64_t n = p->nnz;
  const int64_t nn = n > 0 ? n : 1;
  uint32_t *seg = nullptr, *heads = nullptr;
  int* rows_tmp = nullptr;
  SPM_CUDA_TRY(cudaMallocAsync((void**)&seg, sizeof(uint32_t) * (ceil_div<int64_t>(nn, SEG) + 1), s));
  heads = seg + ceil_div<int64_t>(nn, SEG);
  if (p->lean) SPM_CUDA_TRY(cudaMallocAsync((void**)&rows_tmp, sizeof(int) * nn, s));
  for (int d = 0; d < p->N; ++d) {
    int64_t stride = 0;
    const int* rows = n > 0 ? copy_rows(p, d, rows_tmp, &stride, s) : nullptr;
    partition_copy(p, d, rows, stride, seg, heads, nullptr, s);
  }
  SPM_CUDA_TRY(cudaGetLastError());
  SPM_CUDA_TRY(cudaFreeAsync(seg, s));
  if (rows_tmp) SPM_CUDA_TRY(cudaFreeAsync(rows_tmp, s));
  // a sweep that is captured next must not have to allocate
  return p->als.M ? ensure_als_state(p, s) : SPM_OK;
}

spm_status build_fibre_copies(spmttkrp_plan_s* p, cudaStream_t s);  // fibre_plan.cu

spm_status build_copies(spmttkrp_plan_s* p, const int32_t* const* idx, const float* vals,
                        cudaStream_t s) {
  SPM_TRY(plan_alloc(p, (void**)&p->norm_part, sizeof(double) * NORM_BLOCKS));
  if (record_int4s(p->N) == 1) {
    SPM_TRY(build_copies_t<1>(p, idx, vals, s));
    // the fibre layout is made from the finished record copies (3 modes)
    return p->fibre ? build_fibre_copies(p, s) : SPM_OK;
  }
  return build_copies_t<2>(p, idx, vals, s);
}

}  // namespace spm
