// Tile binning and ordering: device-wide scan, key emission, stable LSD
// radix sort of (key, value) pairs and per-tile ranges.
//
// The compositing order (Eq. 1 composites front to back) is (tile, centre
// depth, surfel index).  It is produced in two levels with the same result
// as one sort of 64-bit (tile << 32 | depth bits) keys: the surfels are
// sorted once by depth (32-bit keys, stable, so ties keep index order), the
// (tile, surfel) instances are emitted in that order, and a stable sort by
// tile id alone (13-16 bits) groups them per tile.
#include "gs2d_internal.cuh"

namespace gs2d {
namespace {

constexpr int kThreads = 256;
constexpr int kItems = 16;  // per thread in one-block scans
constexpr int kWarps = kThreads / 32;
constexpr int kRadixBits = 8;
constexpr int kBins = 1 << kRadixBits;

// Items per thread of the scans and radix passes, by the grid's item bound:
// a small block (1024 items, up to 4M items) spreads a few hundred thousand
// items over all SMs and keeps each block's serial ranking short; larger
// inputs take 2048 (up to 16M) and 4096 items per block, to keep the
// per-block digit counts (and the offsets scan over them) small.
inline int items_per_thread(int64_t n) { return n <= (int64_t(1) << 22) ? 4 : (n <= (int64_t(1) << 24) ? 8 : 16); }
inline int64_t blocks_for(int64_t n) {
  const int64_t ti = (int64_t)kThreads * items_per_thread(n);
  return (n > 0 ? n + ti - 1 : ti) / ti;
}

// Item count: a host bound, lowered to a device-side count when one is given
// (the grid is sized for the bound; blocks past the count do nothing).
__device__ __forceinline__ int64_t item_count(int64_t n_max, const uint32_t* n_dev) {
  if (!n_dev) return n_max;
  const int64_t d = (int64_t)*n_dev;
  return d < n_max ? d : n_max;
}

__device__ __forceinline__ uint32_t warp_incl_scan(uint32_t v) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t t = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += t;
  }
  return v;
}

// Exclusive block scan of one value per thread (256 threads).  Returns the
// exclusive prefix; *total receives the block sum.
__device__ __forceinline__ uint32_t block_excl_scan(uint32_t v, uint32_t* total) {
  __shared__ uint32_t ws[kWarps];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const uint32_t inc = warp_incl_scan(v);
  if (lane == 31) ws[w] = inc;
  __syncthreads();
  if (w == 0) {
    const uint32_t x = lane < kWarps ? ws[lane] : 0u;
    const uint32_t xi = warp_incl_scan(x);
    if (lane < kWarps) ws[lane] = xi - x;
    if (lane == kWarps - 1) *total = xi;
  }
  __syncthreads();
  const uint32_t r = ws[w] + inc - v;
  __syncthreads();
  return r;
}

// Last-block election: every block calls this once, after its thread 0 has
// written the block's result to global memory.  Returns true in the block
// that arrives last, to which all blocks' results are then visible (it reads
// them through L2).  atomicInc wraps the counter back to zero, so it is ready
// for the next launch.
__device__ __forceinline__ bool last_block(uint32_t* done) {
  __shared__ bool last;
  if (threadIdx.x == 0) {
    __threadfence();  // this block's result before its arrival
    last = atomicInc(done, gridDim.x - 1u) == gridDim.x - 1u;
    if (last) __threadfence();
  }
  __syncthreads();
  return last;
}

// Sum of one value per thread over the block (256 threads), in thread 0.
__device__ __forceinline__ uint32_t block_sum(uint32_t v) {
  __shared__ uint32_t ws[kWarps];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if (lane == 0) ws[w] = v;
  __syncthreads();
  uint32_t t = 0;
  if (threadIdx.x == 0)
#pragma unroll
    for (int i = 0; i < kWarps; ++i) t += ws[i];
  return t;
}

// One block: exclusive scan of nb values in place; their sum to *total.
__device__ void block_scan_inplace(uint32_t* __restrict__ v, int nb, uint32_t* __restrict__ total) {
  __shared__ uint32_t tot;
  uint32_t carry = 0;
  for (int base = 0; base < nb; base += kThreads * kItems) {
    // each thread owns kItems consecutive entries of this chunk
    uint32_t x[kItems];
    uint32_t s = 0;
    const int t0 = base + threadIdx.x * kItems;
#pragma unroll
    for (int i = 0; i < kItems; ++i) {
      x[i] = (t0 + i < nb) ? __ldcg(v + t0 + i) : 0u;
      s += x[i];
    }
    uint32_t pre = block_excl_scan(s, &tot) + carry;
#pragma unroll
    for (int i = 0; i < kItems; ++i) {
      if (t0 + i < nb) v[t0 + i] = pre;
      pre += x[i];
    }
    carry += tot;
    __syncthreads();
  }
  if (threadIdx.x == 0 && total) *total = carry;
}

// Block sums of the input; the last block scans them (exclusive, in place)
// and writes the grand total.
template <int kIt>
__global__ void __launch_bounds__(kThreads) scan_reduce(const uint32_t* __restrict__ in, int64_t n_max,
                                                        const uint32_t* __restrict__ n_dev,
                                                        uint32_t* __restrict__ sums,
                                                        uint32_t* __restrict__ total,
                                                        uint32_t* __restrict__ done) {
  const int64_t n = item_count(n_max, n_dev);
  const int64_t base = (int64_t)blockIdx.x * (kThreads * kIt);
  uint32_t x[kIt];
#pragma unroll
  for (int i = 0; i < kIt; ++i) {
    const int64_t k = base + i * kThreads + threadIdx.x;
    x[i] = k < n ? in[k] : 0u;
  }
  uint32_t s = 0;
#pragma unroll
  for (int i = 0; i < kIt; ++i) s += x[i];
  s = block_sum(s);
  if (threadIdx.x == 0) sums[blockIdx.x] = s;
  if (!last_block(done)) return;
  block_scan_inplace(sums, (int)gridDim.x, total);
}

template <int kIt>
__global__ void __launch_bounds__(kThreads) scan_down(const uint32_t* __restrict__ in,
                                                      uint32_t* __restrict__ out, int64_t n_max,
                                                      const uint32_t* __restrict__ n_dev,
                                                      const uint32_t* __restrict__ sums) {
  constexpr int kTI = kThreads * kIt;
  __shared__ uint32_t tile[kTI];
  const int64_t n = item_count(n_max, n_dev);
  const int64_t base = (int64_t)blockIdx.x * kTI;
  if (base >= n) return;
  // coalesced load into shared memory, then each thread scans kIt
  // consecutive entries
  uint32_t x[kIt];
#pragma unroll
  for (int i = 0; i < kIt; ++i) {
    const int64_t k = base + i * kThreads + threadIdx.x;
    x[i] = k < n ? in[k] : 0u;
  }
#pragma unroll
  for (int i = 0; i < kIt; ++i) tile[i * kThreads + threadIdx.x] = x[i];
  __syncthreads();
  uint32_t s = 0;
#pragma unroll
  for (int i = 0; i < kIt; ++i) {
    x[i] = tile[threadIdx.x * kIt + i];
    s += x[i];
  }
  __shared__ uint32_t tot;
  uint32_t pre = block_excl_scan(s, &tot) + sums[blockIdx.x];
#pragma unroll
  for (int i = 0; i < kIt; ++i) {
    tile[threadIdx.x * kIt + i] = pre;
    pre += x[i];
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < kIt; ++i) {
    const int64_t k = base + i * kThreads + threadIdx.x;
    if (k < n) out[k] = tile[i * kThreads + threadIdx.x];
  }
}

// ---- radix sort -----------------------------------------------------------
//
// Per pass: every block counts the digits of its kThreads * kIt keys
// (upsweep); one block per digit scans that digit's counts over the blocks
// (offsets; the counts are stored digit-major, so the scan reads them in
// order); every block then ranks its keys stably (per warp, from ballots of the
// lanes' digit bits; the warps of the block in order) and scatters them
// (downsweep).  Only the blocks that hold items (from the device-side count)
// take part.

// Lanes of the warp whose 9-bit digit equals this lane's: the AND over the
// digit's bits of each bit's ballot (or its complement).
__device__ __forceinline__ uint32_t digit_peers(uint32_t d) {
  uint32_t peers = 0xffffffffu;
#pragma unroll
  for (int b = 0; b < 9; ++b) {
    const uint32_t bl = __ballot_sync(0xffffffffu, (d >> b) & 1u);
    peers &= ((d >> b) & 1u) ? bl : ~bl;
  }
  return peers;
}

template <int kIt>
__global__ void __launch_bounds__(kThreads) radix_upsweep(const uint32_t* __restrict__ keys,
                                                          int64_t n_max, const uint32_t* __restrict__ n_dev,
                                                          int shift, int nbins,
                                                          uint32_t* __restrict__ hist) {
  const int64_t n = item_count(n_max, n_dev);
  if ((int64_t)blockIdx.x * (kThreads * kIt) >= n) return;
  __shared__ uint32_t h[kBins];
  for (int i = threadIdx.x; i < kBins; i += kThreads) h[i] = 0u;
  __syncthreads();
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t base = (int64_t)blockIdx.x * (kThreads * kIt) + w * (32 * kIt);
  const uint32_t mask = (uint32_t)nbins - 1u;
  uint32_t kk[kIt];
#pragma unroll
  for (int it = 0; it < kIt; ++it) {
    const int64_t k = base + it * 32 + lane;
    kk[it] = k < n ? keys[k] : 0u;
  }
#pragma unroll
  for (int it = 0; it < kIt; ++it) {
    const int64_t k = base + it * 32 + lane;
    const bool valid = k < n;
    if (valid) atomicAdd(&h[(kk[it] >> shift) & mask], 1u);
  }
  __syncthreads();
  for (int d = threadIdx.x; d < nbins; d += kThreads) hist[(int64_t)d * gridDim.x + blockIdx.x] = h[d];
}

// Per digit d (one block each): exclusive prefix of the digit's counts over
// the nb_active blocks that hold items, in place, and the digit's total.
__global__ void __launch_bounds__(kThreads) radix_offsets(uint32_t* __restrict__ hist, int nb, int ti,
                                                          int64_t n_max, const uint32_t* __restrict__ n_dev,
                                                          uint32_t* __restrict__ dtot) {
  const int64_t n = item_count(n_max, n_dev);
  const int act = (int)((n + ti - 1) / ti);
  block_scan_inplace(hist + (int64_t)blockIdx.x * nb, act < nb ? act : nb, dtot + blockIdx.x);
}

// gsrc/gout (optional, last pass): gout[dst] = gsrc[value] for every moved
// pair, a gather through the sorted values fused into the scatter.
template <int kIt>
__global__ void __launch_bounds__(kThreads) radix_downsweep(
    const uint32_t* __restrict__ kin, const uint32_t* __restrict__ vin, uint32_t* __restrict__ kout,
    uint32_t* __restrict__ vout, int64_t n_max, const uint32_t* __restrict__ n_dev, int shift, int nbins,
    const uint32_t* __restrict__ offs, const uint32_t* __restrict__ dtot,
    const uint32_t* __restrict__ gsrc, uint32_t* __restrict__ gout) {
  const int64_t n = item_count(n_max, n_dev);
  if ((int64_t)blockIdx.x * (kThreads * kIt) >= n) return;
  __shared__ uint32_t wh[kWarps][kBins];
  __shared__ uint32_t dbase[kBins];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t base = (int64_t)blockIdx.x * (kThreads * kIt) + w * (32 * kIt);
  uint32_t kk[kIt], vv[kIt], pos[kIt];
#pragma unroll
  for (int it = 0; it < kIt; ++it) {
    const int64_t k = base + it * 32 + lane;
    kk[it] = k < n ? kin[k] : 0u;
    vv[it] = k < n ? vin[k] : 0u;
  }
  {
    __shared__ uint32_t tot;
    const uint32_t x = threadIdx.x < nbins ? dtot[threadIdx.x] : 0u;
    dbase[threadIdx.x] = block_excl_scan(x, &tot);
  }
  for (int i = threadIdx.x; i < kWarps * kBins; i += kThreads) (&wh[0][0])[i] = 0u;
  __syncthreads();
  const uint32_t lt = (1u << lane) - 1u;
  const uint32_t mask = (uint32_t)nbins - 1u;
#pragma unroll
  for (int it = 0; it < kIt; ++it) {
    const int64_t k = base + it * 32 + lane;
    const bool valid = k < n;
    const uint32_t d = valid ? ((kk[it] >> shift) & mask) : 0x100u;
    const uint32_t peers = digit_peers(d);
    uint32_t cur = 0u;
    if (valid) cur = wh[w][d];
    __syncwarp();
    if (valid && lane == (31 - __clz(peers))) wh[w][d] = cur + (uint32_t)__popc(peers);
    __syncwarp();
    pos[it] = valid ? cur + (uint32_t)__popc(peers & lt) : 0xFFFFFFFFu;
  }
  __syncthreads();
  for (int d = threadIdx.x; d < nbins; d += kThreads) {
    uint32_t run = dbase[d] + offs[(int64_t)d * gridDim.x + blockIdx.x];
#pragma unroll
    for (int ww = 0; ww < kWarps; ++ww) {
      const uint32_t t = wh[ww][d];
      wh[ww][d] = run;
      run += t;
    }
  }
  __syncthreads();
#pragma unroll
  for (int it = 0; it < kIt; ++it) {
    if (pos[it] == 0xFFFFFFFFu) continue;
    const uint32_t d = (kk[it] >> shift) & mask;
    const uint32_t dst = wh[w][d] + pos[it];
    kout[dst] = kk[it];
    vout[dst] = vv[it];
    if (gout) gout[dst] = gsrc[vv[it]];
  }
}

// ---- few items ------------------------------------------------------------
//
// Up to kSmallMax items one block does a whole scan, or all passes of a sort:
// each launch costs a small scene more than its work.  A view of 2000 to 4096
// surfels at 128 x 128 with loss and backward: 345 us with three launches a
// pass (15 to 18 for its two sorts) and two a scan, 289 so.  With four times
// as many items a thread, up to 16384 in all, one SM's ranking of them eats the
// launches: 6000 surfels 352 against 357 us, 10000 396 and 394, 16000 432 and 414.
constexpr int kSmallThreads = 1024;
constexpr int kSmallWarps = kSmallThreads / 32;
constexpr int kSmallIt = 4;
constexpr int kSmallMax = kSmallIt * kSmallThreads;

// Exclusive scan of one value per thread (1024 threads).
__device__ __forceinline__ uint32_t small_excl_scan(uint32_t v, uint32_t* total) {
  __shared__ uint32_t ws[kSmallWarps];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const uint32_t inc = warp_incl_scan(v);
  if (lane == 31) ws[w] = inc;
  __syncthreads();
  if (w == 0) {
    const uint32_t x = ws[lane], xi = warp_incl_scan(x);
    ws[lane] = xi - x;
    if (lane == 31) *total = xi;
  }
  __syncthreads();
  return ws[w] + inc - v;
}

__global__ void __launch_bounds__(kSmallThreads) scan_small(const uint32_t* in, uint32_t* out, int64_t n_max,
                                                            const uint32_t* __restrict__ n_dev,
                                                            uint32_t* __restrict__ total) {
  constexpr int kIt = kSmallIt;
  __shared__ uint32_t tot;
  const int n = (int)item_count(n_max, n_dev);
  const int t0 = (int)threadIdx.x * kIt;
  uint32_t x[kIt], s = 0;
#pragma unroll
  for (int i = 0; i < kIt; ++i) {
    x[i] = t0 + i < n ? in[t0 + i] : 0u;
    s += x[i];
  }
  uint32_t pre = small_excl_scan(s, &tot);
#pragma unroll
  for (int i = 0; i < kIt; ++i) {
    if (t0 + i < n) out[t0 + i] = pre;
    pre += x[i];
  }
  if (total && threadIdx.x == 0) *total = tot;
}

struct SmallSort {
  uint32_t k[kSmallMax], v[kSmallMax];
  uint16_t wh[kSmallWarps][kBins];  // per warp and digit: counts, then the warp's start within the digit
  uint32_t dbase[kBins];
  uint32_t tot;
};

// All passes, in place: the items stay in registers between a pass's ranking
// (as in radix_downsweep) and its exchange through shared memory.
__global__ void __launch_bounds__(kSmallThreads) radix_small(uint32_t* keys, uint32_t* vals, int64_t n_max,
                                                             const uint32_t* __restrict__ n_dev, int bits,
                                                             const uint32_t* __restrict__ gsrc,
                                                             uint32_t* __restrict__ gout) {
  extern __shared__ __align__(16) unsigned char small_smem[];
  constexpr int kIt = kSmallIt;
  SmallSort& S = *reinterpret_cast<SmallSort*>(small_smem);
  const int n = (int)item_count(n_max, n_dev);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int i0 = w * (32 * kIt) + lane;
  const uint32_t lt = (1u << lane) - 1u;
  uint32_t kk[kIt], vv[kIt];
#pragma unroll
  for (int it = 0; it < kIt; ++it) {
    const int i = i0 + it * 32;
    kk[it] = i < n ? keys[i] : 0u;
    vv[it] = i < n ? vals[i] : 0u;
  }
  for (int shift = 0; shift < bits; shift += kRadixBits) {
    const uint32_t mask = (1u << min(bits - shift, kRadixBits)) - 1u;
    for (int i = threadIdx.x; i < kSmallWarps * kBins / 2; i += kSmallThreads)
      reinterpret_cast<uint32_t*>(&S.wh[0][0])[i] = 0u;
    __syncthreads();
    uint32_t pos[kIt];
#pragma unroll
    for (int it = 0; it < kIt; ++it) {
      const bool valid = i0 + it * 32 < n;
      const uint32_t d = valid ? (kk[it] >> shift) & mask : 0x100u;
      const uint32_t peers = digit_peers(d);
      uint32_t cur = 0u;
      if (valid) cur = S.wh[w][d];
      __syncwarp();
      if (valid && lane == 31 - __clz(peers)) S.wh[w][d] = (uint16_t)(cur + (uint32_t)__popc(peers));
      __syncwarp();
      pos[it] = cur + (uint32_t)__popc(peers & lt);
    }
    __syncthreads();
    uint32_t run = 0u;
    if (threadIdx.x < kBins)
      for (int ww = 0; ww < kSmallWarps; ++ww) {
        const uint32_t c = S.wh[ww][threadIdx.x];
        S.wh[ww][threadIdx.x] = (uint16_t)run;
        run += c;
      }
    const uint32_t base = small_excl_scan(run, &S.tot);
    if (threadIdx.x < kBins) S.dbase[threadIdx.x] = base;
    __syncthreads();
#pragma unroll
    for (int it = 0; it < kIt; ++it) {
      if (i0 + it * 32 >= n) continue;
      const uint32_t d = (kk[it] >> shift) & mask;
      const uint32_t dst = S.dbase[d] + S.wh[w][d] + pos[it];
      S.k[dst] = kk[it];
      S.v[dst] = vv[it];
    }
    __syncthreads();
#pragma unroll
    for (int it = 0; it < kIt; ++it) {
      const int i = i0 + it * 32;
      if (i >= n) continue;
      kk[it] = S.k[i];
      vv[it] = S.v[i];
    }
  }
#pragma unroll
  for (int it = 0; it < kIt; ++it) {
    const int i = i0 + it * 32;
    if (i >= n) continue;
    keys[i] = kk[it];
    vals[i] = vv[it];
    if (gout) gout[i] = gsrc[vv[it]];
  }
}

__global__ void gather_counts_kernel(const uint32_t* __restrict__ order,
                                     const uint32_t* __restrict__ tcount, uint32_t* __restrict__ out,
                                     int64_t n_max, const uint32_t* __restrict__ n_dev) {
  const int64_t n = item_count(n_max, n_dev);
  const int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (r < n) out[r] = tcount[order[r]];
}

// Instances of surfel order[r] at offsets offs[r]..: for every tile row of
// its rectangle, the tile columns its footprint reaches (the same row rule,
// on the same stored doubles, that counted them in the preprocess), row by
// row, left to right.  A warp takes 32 consecutive candidates, whose instances
// are one run of the output.  It moves their footprints into shared memory
// (a lane's own loads of its 56 bytes would touch 32 cache lines each), spreads
// their tile rows over its lanes, then the rows' tiles, so that neither a long
// footprint nor a long row keeps one lane busy while the others wait, and
// consecutive lanes write consecutive instances.
//
// kMask: the tile index takes the key's lower 16 bits and the upper 16 hold
// the mask of the tile's 4 x 4 pixel blocks that the footprint can reach (the
// row rule on the tile row's four bands of four pixel rows, found once per
// row of tiles).  The sort carries it along.  Made per sorted instance
// instead, from a gather of the footprints, the masks alone took 287 us of
// four 900p views of 4M surfels and 354 us of a 4K view of 8M; emission and
// ranges together went from 623 to 466 and from 563 to 310 us there (1M
// surfels at 900p: 65 to 51).  What bounds it is the latency of the footprints'
// gather and of the steps between a row's tiles and their places (with
// searches by shuffles instead of marked starts 567 and 369 us); four blocks
// per SM, three and five measured 685 and 478, 446 and 321.
__device__ __forceinline__ uint32_t band_nibble(uint32_t blocks, int tx) {
  // blocks: first and last of the band's 4-pixel block columns (16 bits each)
  const int lo = max((int)(blocks & 0xffffu) - 4 * tx, 0), hi = min((int)(blocks >> 16) - 4 * tx, 3);
  return lo <= hi ? (15u >> (3 - hi)) & (15u << lo) : 0u;
}

struct EmitSmem {
  uint2 geom[32 * sizeof(RowGeom) / sizeof(uint2)];
  uint4 cand[32];    // candidates with rows, in order: surfel, first tile row - first flattened row, lane
  uint4 row[32][2];  // tile rows with tiles, in order: key of flattened tile 0, surfel, tile column of it; bands
};

template <bool kMask>
__device__ __forceinline__ void emit_warp(int64_t r, int64_t n, int lane, const uint32_t* __restrict__ order,
                                          const uint32_t* __restrict__ offs, const uint32_t* __restrict__ counts,
                                          const uint2* __restrict__ rect, const RowGeom* __restrict__ geom,
                                          float rf, int tiles_x, EmitSmem& sm, uint32_t* __restrict__ keys,
                                          uint32_t* __restrict__ vals) {
  constexpr unsigned kFull = 0xffffffffu;
  constexpr int kPieces = (int)(sizeof(RowGeom) / sizeof(uint2));
  const uint32_t lt = (1u << lane) - 1u, upto = lt | (1u << lane);
  const bool valid = r < n && counts[r] > 0u;
  uint32_t s = 0xffffffffu;
  int ty0 = 0, nrows = 0;
  if (valid) {
    s = order[r];
    const uint2 rc = rect[s];
    ty0 = (int)(rc.x >> 16);
    nrows = (int)(rc.y >> 16) - ty0;
  }
  uint32_t out = __shfl_sync(kFull, r < n ? offs[r] : 0u, 0);  // the run's next position
#pragma unroll
  for (int p = 0; p < kPieces; ++p) {
    const int k = p * 32 + lane, row = k / kPieces;
    const uint32_t sr = __shfl_sync(kFull, s, row);
    if (sr != 0xffffffffu) sm.geom[k] = reinterpret_cast<const uint2*>(geom + sr)[k - row * kPieces];
  }
  // exclusive prefix of the row counts over the warp: lane i's rows are
  // flattened rows [first, first + nrows)
  int incl = nrows;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(kFull, incl, o);
    if (lane >= o) incl += t;
  }
  const int first = incl - nrows;
  const int total = __shfl_sync(kFull, incl, 31);
  const uint32_t has = __ballot_sync(kFull, nrows > 0);
  if (nrows > 0) sm.cand[__popc(has & lt)] = make_uint4(s, (uint32_t)(ty0 - first), (uint32_t)lane, 0u);
  __syncwarp();
  int before = -1;  // owners of earlier chunks' rows, less one
  for (int c0 = 0; c0 < total; c0 += 32) {
    const int j = c0 + lane;
    // a row's owner: the last candidate whose first row is at or before it
    const uint32_t heads =
        __reduce_or_sync(kFull, nrows > 0 && first >= c0 && first < c0 + 32 ? 1u << (first - c0) : 0u);
    const uint4 cd = sm.cand[before + __popc(heads & upto)];
    before += __popc(heads);
    const int ty = (int)cd.y + j;
    int a = 0, b = 0;
    uint32_t band[4] = {0xffffu, 0xffffu, 0xffffu, 0xffffu};  // none
    if (j < total) {
      const RowGeom g = reinterpret_cast<const RowGeom*>(sm.geom)[cd.z];
      if (!row_tiles(g, ty, rf, &a, &b)) a = b = 0;
      if constexpr (kMask) {
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int ja = ty * kTile + 4 * q;
          int ilo, ihi;
          if (band_pixels(g, ja, ja + 3, rf, &ilo, &ihi)) band[q] = (uint32_t)(ilo >> 2) | ((uint32_t)(ihi >> 2) << 16);
        }
      }
    }
    // the chunk's tiles: this row has [sx, sx + b - a) of them
    int sc = b - a;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int x = __shfl_up_sync(kFull, sc, o);
      if (lane >= o) sc += x;
    }
    const int sx = sc - (b - a);
    const int tiles = __shfl_sync(kFull, sc, 31);
    const uint32_t some = __ballot_sync(kFull, b > a);
    if (b > a) {
      const int q = __popc(some & lt);
      sm.row[q][0] = make_uint4((uint32_t)(ty * tiles_x + a - sx), cd.x, (uint32_t)(a - sx), 0u);
      if constexpr (kMask) sm.row[q][1] = make_uint4(band[0], band[1], band[2], band[3]);
    }
    __syncwarp();
    int rows = -1;  // rows that start in earlier windows, less one
    for (int t0 = 0; t0 < tiles; t0 += 32) {
      const int t = t0 + lane;
      const uint32_t starts = __reduce_or_sync(kFull, b > a && sx >= t0 && sx < t0 + 32 ? 1u << (sx - t0) : 0u);
      const int q = rows + __popc(starts & upto);
      rows += __popc(starts);
      if (t >= tiles) continue;
      const uint4 rw = sm.row[q][0];
      uint32_t key = rw.x + (uint32_t)t;
      if constexpr (kMask) {
        const uint4 bd = sm.row[q][1];
        const int tx = (int)rw.z + t;
        uint32_t m = 0u;
#pragma unroll
        for (int h = 0; h < 4; ++h) {
          const uint32_t nib = band_nibble(h == 0 ? bd.x : (h == 1 ? bd.y : (h == 2 ? bd.z : bd.w)), tx);
          // block columns 0, 1 and 2, 3 of block row h
          m |= ((nib & 3u) | ((nib & 12u) << 2)) << (8 * (h >> 1) + 2 * (h & 1));
        }
        key |= m << 16;
      }
      keys[out + (uint32_t)t] = key;
      vals[out + (uint32_t)t] = rw.y;
    }
    out += (uint32_t)tiles;
    __syncwarp();  // before the next chunk's rows, the next candidates' footprints
  }
}

template <bool kMask>
__global__ void __launch_bounds__(256, 4) emit_kernel(const uint32_t* __restrict__ order,
                                                   const uint32_t* __restrict__ offs,
                                                   const uint32_t* __restrict__ counts,
                                                   const uint2* __restrict__ rect,
                                                   const RowGeom* __restrict__ geom, float rf, int64_t n_max,
                                                   const uint32_t* __restrict__ n_dev, int tiles_x,
                                                   uint32_t* __restrict__ keys, uint32_t* __restrict__ vals) {
  __shared__ EmitSmem stage[8];
  const int64_t n = item_count(n_max, n_dev);
  const int lane = threadIdx.x & 31;
  // grid-stride over warps of 32 candidates (the grid is sized for the
  // resident CTAs, the count is known on the device only)
  for (int64_t r0 = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); r0 < n;
       r0 += (int64_t)gridDim.x * blockDim.x)
    emit_warp<kMask>(r0 + lane, n, lane, order, offs, counts, rect, geom, rf, tiles_x, stage[threadIdx.x >> 5], keys,
                     vals);
}

// Four sorted instances a thread: the ends of their tiles' ranges, and the
// masks out of their keys.  Bound by the keys' and masks' traffic.
__global__ void __launch_bounds__(256) ranges_of_keys(const uint32_t* __restrict__ keys, int64_t K,
                                                      int2* __restrict__ ranges, uint16_t* __restrict__ masks) {
  const int64_t i0 = 4 * ((int64_t)blockIdx.x * blockDim.x + threadIdx.x);
  if (i0 >= K) return;
  uint32_t k[6];  // the four and their neighbours
  const int m = (int)min((int64_t)4, K - i0);
  if (m == 4) {
    const uint4 v = *reinterpret_cast<const uint4*>(keys + i0);
    k[1] = v.x; k[2] = v.y; k[3] = v.z; k[4] = v.w;
    *reinterpret_cast<uint2*>(masks + i0) = make_uint2((v.x >> 16) | (v.y & 0xffff0000u), (v.z >> 16) | (v.w & 0xffff0000u));
  } else {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      k[q + 1] = q < m ? keys[i0 + q] : 0u;
      if (q < m) masks[i0 + q] = (uint16_t)(k[q + 1] >> 16);
    }
  }
  k[0] = i0 > 0 ? keys[i0 - 1] : 0u;
  k[5] = i0 + 4 < K ? keys[i0 + 4] : 0u;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int64_t i = i0 + q;
    const uint32_t t = k[q + 1] & 0xffffu;
    if (q >= m) continue;
    if (i == 0 || (k[q] & 0xffffu) != t) ranges[t].x = (int)i;
    if (i == K - 1 || (k[q + 2] & 0xffffu) != t) ranges[t].y = (int)(i + 1);
  }
}

// Keys without masks: one thread per sorted instance, the mask from the
// footprint as emit_warp<true> makes it.
__global__ void __launch_bounds__(256) ranges_kernel(const uint32_t* __restrict__ keys,
                                                     const uint32_t* __restrict__ vals, int64_t K,
                                                     int2* __restrict__ ranges, const RowGeom* __restrict__ geom,
                                                     float rf, int tiles_x, int H, uint16_t* __restrict__ masks) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= K) return;
  const uint32_t t = keys[i];
  const RowGeom g = geom[vals[i]];
  if (i == 0 || keys[i - 1] != t) ranges[t].x = (int)i;
  if (i == K - 1 || keys[i + 1] != t) ranges[t].y = (int)(i + 1);
  const int tx0 = (int)(t % (uint32_t)tiles_x) * kTile, ty0 = (int)(t / (uint32_t)tiles_x) * kTile;
  uint32_t m = 0u;
#pragma unroll
  for (int b = 0; b < 4; ++b) {
    const int ja = ty0 + 4 * b;
    int ilo, ihi;
    if (ja >= H || !band_pixels(g, ja, min(ja + 3, H - 1), rf, &ilo, &ihi)) continue;
#pragma unroll
    for (int c = 0; c < 4; ++c)
      if (ilo <= tx0 + 4 * c + 3 && ihi >= tx0 + 4 * c)
        m |= 1u << (4 * ((c >> 1) | (b & 2)) + ((c & 1) | ((b & 1) << 1)));
  }
  masks[i] = (uint16_t)m;
}

// Tiles ordered by list length, longest first (by octave of the length;
// order within an octave is arbitrary): launching the blends in this order
// starts the longest tiles first, so the last wave is short ones.  Results
// do not depend on the order.  One block; the octaves are staged in shared
// memory (up to kMaxOrderTiles tiles).
constexpr int kMaxOrderTiles = 40960;
__global__ void __launch_bounds__(1024) tile_order_kernel(const int2* __restrict__ ranges, int ntiles,
                                                          uint32_t* __restrict__ order) {
  __shared__ uint8_t oct[kMaxOrderTiles];
  __shared__ uint32_t cnt[32], cur[32];
  const int lane = threadIdx.x & 31;
  if (threadIdx.x < 32) cnt[threadIdx.x] = 0u;
  __syncthreads();
  // per warp and octave one shared-memory atomic (lanes of the same octave
  // are counted together): a few octaves hold most tiles
  for (int t0 = threadIdx.x - lane; t0 < ntiles; t0 += blockDim.x) {
    const int t = t0 + lane;
    const bool valid = t < ntiles;
    uint32_t o = 32u;
    if (valid) {
      const int2 r = ranges[t];
      o = (uint32_t)__clz((uint32_t)(r.y - r.x) | 1u);  // 31 - octave: longest first
      oct[t] = (uint8_t)o;
    }
    const uint32_t peers = __match_any_sync(0xffffffffu, o);
    if (valid && lane == 31 - __clz(peers)) atomicAdd(&cnt[o], (uint32_t)__popc(peers));
  }
  __syncthreads();
  if (threadIdx.x < 32) {
    // exclusive scan of the 32 bucket counts in one warp
    const uint32_t c = cnt[threadIdx.x];
    uint32_t v = c;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t u = __shfl_up_sync(0xffffffffu, v, d);
      if ((int)threadIdx.x >= d) v += u;
    }
    cur[threadIdx.x] = v - c;
  }
  __syncthreads();
  for (int t0 = threadIdx.x - lane; t0 < ntiles; t0 += blockDim.x) {
    const int t = t0 + lane;
    const bool valid = t < ntiles;
    const uint32_t o = valid ? (uint32_t)oct[t] : 32u;
    const uint32_t peers = __match_any_sync(0xffffffffu, o);
    const int leader = 31 - __clz(peers);
    uint32_t base = 0u;
    if (valid && lane == leader) base = atomicAdd(&cur[o], (uint32_t)__popc(peers));
    base = __shfl_sync(0xffffffffu, base, leader);
    if (valid) order[base + (uint32_t)__popc(peers & ((1u << lane) - 1u))] = (uint32_t)t;
  }
}

}  // namespace

// block sums, then the last-block counter
size_t scan_tmp_words(int64_t n) { return (size_t)blocks_for(n) + 2; }

cudaError_t launch_scan(const uint32_t* in, uint32_t* out, int64_t n, uint32_t* total_dev,
                        uint32_t* tmp, cudaStream_t st, const uint32_t* n_dev) {
  if (n <= 0) {
    return total_dev ? cudaMemsetAsync(total_dev, 0, sizeof(uint32_t), st) : cudaSuccess;
  }
  ProfScope ps(kProfSort, st);
  if (n <= kSmallMax) {
    count_launch();
    scan_small<<<1, kSmallThreads, 0, st>>>(in, out, n, n_dev, total_dev);
    return cudaGetLastError();
  }
  const unsigned nb = (unsigned)blocks_for(n);
  uint32_t* done = tmp + nb + 1;
  cudaError_t e = cudaMemsetAsync(done, 0, sizeof(uint32_t), st);
  if (e != cudaSuccess) return e;
  count_launch(2);
  switch (items_per_thread(n)) {
    case 4:
      scan_reduce<4><<<nb, kThreads, 0, st>>>(in, n, n_dev, tmp, total_dev, done);
      scan_down<4><<<nb, kThreads, 0, st>>>(in, out, n, n_dev, tmp);
      break;
    case 8:
      scan_reduce<8><<<nb, kThreads, 0, st>>>(in, n, n_dev, tmp, total_dev, done);
      scan_down<8><<<nb, kThreads, 0, st>>>(in, out, n, n_dev, tmp);
      break;
    default:
      scan_reduce<16><<<nb, kThreads, 0, st>>>(in, n, n_dev, tmp, total_dev, done);
      scan_down<16><<<nb, kThreads, 0, st>>>(in, out, n, n_dev, tmp);
      break;
  }
  return cudaGetLastError();
}

// digit-major counts (kBins rows of one word per block), then the digit totals
size_t radix_tmp_words(int64_t n) { return (size_t)blocks_for(n) * kBins + kBins; }

namespace {
template <int kIt>
void radix_pass(const uint32_t* ki, const uint32_t* vi, uint32_t* ko, uint32_t* vo, int64_t n,
                const uint32_t* n_dev, int shift, int nbins, unsigned nb, uint32_t* hist, uint32_t* dtot,
                const uint32_t* gsrc, uint32_t* gout, cudaStream_t st) {
  radix_upsweep<kIt><<<nb, kThreads, 0, st>>>(ki, n, n_dev, shift, nbins, hist);
  radix_offsets<<<nbins, kThreads, 0, st>>>(hist, (int)nb, kThreads * kIt, n, n_dev, dtot);
  radix_downsweep<kIt><<<nb, kThreads, 0, st>>>(ki, vi, ko, vo, n, n_dev, shift, nbins, hist, dtot, gsrc, gout);
}

cudaError_t sort_small(uint32_t* keys, uint32_t* vals, int64_t n, const uint32_t* n_dev, int bits,
                       const uint32_t* gsrc, uint32_t* gout, cudaStream_t st) {
  const int smem = (int)sizeof(SmallSort);
  const cudaError_t e = cudaFuncSetAttribute(radix_small, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  count_launch();
  radix_small<<<1, kSmallThreads, smem, st>>>(keys, vals, n, n_dev, bits, gsrc, gout);
  return cudaGetLastError();
}
}  // namespace

cudaError_t radix_sort_pairs(uint32_t* keys, uint32_t* vals, uint32_t* keys_alt,
                             uint32_t* vals_alt, int64_t n, int bits, uint32_t* tmp,
                             uint32_t** keys_out, uint32_t** vals_out, cudaStream_t st,
                             const uint32_t* n_dev, const uint32_t* gsrc, uint32_t* gout) {
  *keys_out = keys;
  *vals_out = vals;
  if (n <= 1 || bits <= 0) {
    // no pass to fuse the gather into
    return gout ? launch_gather_counts(vals, gsrc, gout, n, st, n_dev) : cudaSuccess;
  }
  ProfScope ps(kProfSort, st);
  if (n <= kSmallMax) return sort_small(keys, vals, n, n_dev, bits, gsrc, gout, st);
  const unsigned nb = (unsigned)blocks_for(n);
  const int it = items_per_thread(n);
  uint32_t* hist = tmp;
  uint32_t* dtot = tmp + (size_t)nb * kBins;
  uint32_t *ki = keys, *vi = vals, *ko = keys_alt, *vo = vals_alt;
  for (int shift = 0; shift < bits; shift += kRadixBits) {
    const int pb = bits - shift < kRadixBits ? bits - shift : kRadixBits;
    const int nbins = 1 << pb;
    const bool last = shift + kRadixBits >= bits;
    const uint32_t* gs = last ? gsrc : nullptr;
    uint32_t* go = last ? gout : nullptr;
    count_launch(3);
    if (it == 4) radix_pass<4>(ki, vi, ko, vo, n, n_dev, shift, nbins, nb, hist, dtot, gs, go, st);
    else if (it == 8) radix_pass<8>(ki, vi, ko, vo, n, n_dev, shift, nbins, nb, hist, dtot, gs, go, st);
    else radix_pass<16>(ki, vi, ko, vo, n, n_dev, shift, nbins, nb, hist, dtot, gs, go, st);
    uint32_t* t = ki; ki = ko; ko = t;
    t = vi; vi = vo; vo = t;
  }
  *keys_out = ki;
  *vals_out = vi;
  return cudaGetLastError();
}

cudaError_t launch_gather_counts(const uint32_t* order, const uint32_t* tcount, uint32_t* out,
                                 int64_t n, cudaStream_t st, const uint32_t* n_dev) {
  if (n <= 0) return cudaSuccess;
  ProfScope ps(kProfSort, st);
  count_launch();
  gather_counts_kernel<<<div_up(n, 256), 256, 0, st>>>(order, tcount, out, n, n_dev);
  return cudaGetLastError();
}

// Masks in the keys wherever the tile indices leave them 16 bits (images of up
// to 16.7 million pixels) and the 4-pixel block columns fit 16 bits.
static bool masks_in_keys(const CamDev& cam) {
  return (int64_t)cam.tiles_x * cam.tiles_y <= 65536 && cam.tiles_x <= 16384;
}

cudaError_t launch_emit(const uint32_t* order, const uint32_t* offs, const uint32_t* counts,
                        const uint2* rect, const RowGeom* geom, float rf, int64_t n, const CamDev& cam,
                        uint32_t* keys, uint32_t* vals, cudaStream_t st, const uint32_t* n_dev) {
  if (n <= 0) return cudaSuccess;
  ProfScope ps(kProfSort, st);
  count_launch();
  // at most two waves (the count of candidates is on the device; the bound n
  // is usually several times larger)
  const unsigned resident = 8u * sm_count();
  const unsigned blocks = div_up(n, 256) < resident ? div_up(n, 256) : resident;
  if (masks_in_keys(cam))
    emit_kernel<true><<<blocks, 256, 0, st>>>(order, offs, counts, rect, geom, rf, n, n_dev, cam.tiles_x, keys, vals);
  else
    emit_kernel<false><<<blocks, 256, 0, st>>>(order, offs, counts, rect, geom, rf, n, n_dev, cam.tiles_x, keys, vals);
  return cudaGetLastError();
}

cudaError_t launch_ranges(const uint32_t* keys, const uint32_t* vals, int64_t K, int2* ranges, int ntiles,
                          const RowGeom* geom, float rf, const CamDev& cam, uint16_t* masks, cudaStream_t st) {
  ProfScope ps(kProfSort, st);
  cudaError_t e = cudaMemsetAsync(ranges, 0, sizeof(int2) * (size_t)ntiles, st);
  if (e != cudaSuccess || K <= 0) return e;
  count_launch();
  if (masks_in_keys(cam))
    ranges_of_keys<<<div_up((K + 3) / 4, 256), 256, 0, st>>>(keys, K, ranges, masks);
  else
    ranges_kernel<<<div_up(K, 256), 256, 0, st>>>(keys, vals, K, ranges, geom, rf, cam.tiles_x, cam.H, masks);
  return cudaGetLastError();
}

bool tile_order_supported(int ntiles) { return ntiles > 0 && ntiles <= kMaxOrderTiles; }

cudaError_t launch_tile_order(const int2* ranges, int ntiles, uint32_t* order, cudaStream_t st) {
  if (!tile_order_supported(ntiles)) return cudaSuccess;
  ProfScope ps(kProfSort, st);
  count_launch();
  tile_order_kernel<<<1, 1024, 0, st>>>(ranges, ntiles, order);
  return cudaGetLastError();
}

}  // namespace gs2d
