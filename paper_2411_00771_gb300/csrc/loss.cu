// Photometric and depth losses with their adjoints (Sec. 3.1: L1 + D-SSIM;
// Sec. 3.2: L1 on inverse depth).
//
// Kernel 1, per 32 x 54 tile and colour channel: stages a 42 x 64 halo of
// the render and the target in shared memory, forms the five windowed
// moments (mu_x, mu_y, E[x^2], E[y^2], E[xy]) with the separable 11-tap
// Gaussian (zero padded), the SSIM map and its partials with respect to
// mu_x, E[x^2] and E[xy]; the partials go to scratch, the map and |x - y| to
// per-block sums.  Kernel 2 blurs the three partial maps again (the window
// is symmetric, so the adjoint of the windowed sum is the same windowed sum)
// and writes the adjoint planes of the weighted SSIM term, the weighted L1
// term and their sum, plus the inverse-depth adjoint.  A last one-block
// kernel reduces the per-block sums in double.
//
// Both blurs slide the window in registers: a thread of the horizontal pass
// reads 18 inputs of one row and produces 8 outputs, a thread of the
// vertical pass reads 17 rows of one column and produces 7, so each staged
// value is read from shared memory a few times instead of 22; two maps at a
// time go through the packed FP32 instructions.  What bounds both kernels is
// the shared-memory and FMA pipes together (57 and 48 % busy) and the barriers
// between the passes.  The tile's height makes one horizontal item of each
// thread: at 32 x 32, 168 of 256 threads had one and the others waited, and a
// halo value served 0.58 outputs instead of 0.64.  The horizontal sums take the
// halo's place, so that four (forward) and five blocks fit an SM.  1600 x 900, forward and
// backward kernel, us: one map at a time 47.5 and 48; two, 32 x 32 tiles 42.7
// and 47; 32 x 54 39 and 46 (the backward with four and three blocks an SM
// 51 and 60).
#include <math.h>

#include <mutex>
#include <string>

#include "gs2d_internal.cuh"

namespace gs2d {
namespace {

constexpr int kTW = 32, kTH = 54;    // output tile
constexpr int kR = 5;                // window radius (11 taps)
constexpr int kHaloW = kTW + 2 * kR; // 42
constexpr int kHaloH = kTH + 2 * kR; // 64
constexpr int kTaps = 2 * kR + 1;
constexpr int kThr = 256;
constexpr int kHS = 8;               // outputs per horizontal item
constexpr int kVS = 7;               // outputs per vertical item
constexpr int kSX = kHaloW + 1;      // odd row stride of the staged halo
constexpr int kSH = kTW + 1;         // row stride of the horizontal sums
constexpr int kSumH = (kThr / kTW) * kVS + 2 * kR;  // rows the vertical items read (the last two: not used)
static_assert(kHaloH * (kTW / kHS) == kThr, "one horizontal item per thread");
static_assert((kThr / kTW) * kVS >= kTH && kSumH * kSH <= kHaloH * kSX, "vertical items cover the tile; sums fit the halo");

struct Gauss {
  float w[kTaps];
};

// Stage a kHaloW x kHaloH window (top-left at (ox, oy)) of NP planes of a
// W x H image, zero outside the image, the first two as pairs; all loads of a
// thread are issued before the first store.  Thread t takes column t % kHaloW
// of rows t / kHaloW, + kStageRows, ...: its index arithmetic is done once.
constexpr int kStageRows = kThr / kHaloW;                          // 6
constexpr int kStageIt = (kHaloH + kStageRows - 1) / kStageRows;   // 11
template <int NP>
struct Planes {
  const float* p[NP];
};
template <int NP>
__device__ __forceinline__ void stage_halo(float2 (*pair)[kSX], float (*third)[kSX], Planes<NP> src, int W, int H,
                                           int ox, int oy) {
  const int r0 = threadIdx.x / kHaloW, hx = threadIdx.x - r0 * kHaloW;
  if (r0 >= kStageRows) return;
  const int gx = ox + hx;
  const bool inx = gx >= 0 && gx < W;
  float v[NP][kStageIt];
#pragma unroll
  for (int k = 0; k < kStageIt; ++k) {
    const int hy = r0 + k * kStageRows, gy = oy + hy;
    const bool in = inx && hy < kHaloH && gy >= 0 && gy < H;
#pragma unroll
    for (int q = 0; q < NP; ++q) v[q][k] = in ? src.p[q][(size_t)gy * W + gx] : 0.f;
  }
#pragma unroll
  for (int k = 0; k < kStageIt; ++k) {
    const int hy = r0 + k * kStageRows;
    if (hy < kHaloH) {
      pair[hy][hx] = make_float2(v[0][k], v[1][k]);
      if constexpr (NP == 3) third[hy][hx] = v[2][k];
    }
  }
}

// out[i] = sum_k w[k] in[i + k] for kHS (or kVS) consecutive outputs, with
// the inputs already in registers; of one map, or of two at a time on the
// packed FP32 instructions (the same operations in the same order per map).
template <int NO>
__device__ __forceinline__ void slide(const float* in, const Gauss& g, float* o) {
#pragma unroll
  for (int j = 0; j < NO + kTaps - 1; ++j)
#pragma unroll
    for (int i = 0; i < NO; ++i) {
      if (j == i) o[i] = g.w[0] * in[j];
      else if (j - i > 0 && j - i < kTaps) o[i] = fmaf(g.w[j - i], in[j], o[i]);
    }
}
template <int NO>
__device__ __forceinline__ void slide(const float2* in, const Gauss& g, float2* o) {
#pragma unroll
  for (int j = 0; j < NO + kTaps - 1; ++j)
#pragma unroll
    for (int i = 0; i < NO; ++i) {
      const float w = g.w[j - i >= 0 && j - i < kTaps ? j - i : 0];
      if (j == i) o[i] = __fmul2_rn(make_float2(w, w), in[j]);
      else if (j - i > 0 && j - i < kTaps) o[i] = __ffma2_rn(make_float2(w, w), in[j], o[i]);
    }
}

__global__ void __launch_bounds__(kThr, 3) ssim_fwd_kernel(int W, int H, const float* __restrict__ out,
                                                        const float* __restrict__ tgt, Gauss g,
                                                        float* __restrict__ part,
                                                        float* __restrict__ bsum) {
  __shared__ float2 sxy[kHaloH][kSX];
  __shared__ float2 h2[kSumH][kSH];  // moments (x^2, y^2)
  __shared__ float h3[kSumH][kSH];   // x y
  float2 (*const h1)[kSH] = reinterpret_cast<float2 (*)[kSH]>(sxy);  // (x, y), in the halo's place
  const int c = blockIdx.z;
  const size_t HW = (size_t)W * H;
  const int ox = blockIdx.x * kTW - kR, oy = blockIdx.y * kTH - kR;
  const int t = threadIdx.x;
  stage_halo<2>(sxy, nullptr, Planes<2>{{out + c * HW, tgt + c * HW}}, W, H, ox, oy);
  __syncthreads();
  // horizontal pass over all halo rows: item = (row, 8-column segment)
  {
    const int r = t % kHaloH, c0 = (t / kHaloH) * kHS;
    float2 in[kHS + kTaps - 1], o[kHS];
#pragma unroll
    for (int j = 0; j < kHS + kTaps - 1; ++j) in[j] = sxy[r][c0 + j];
    __syncthreads();  // the halo is read
    slide<kHS>(in, g, o);
#pragma unroll
    for (int i = 0; i < kHS; ++i) h1[r][c0 + i] = o[i];
    float xy[kHS + kTaps - 1], p[kHS];
#pragma unroll
    for (int j = 0; j < kHS + kTaps - 1; ++j) {
      xy[j] = in[j].x * in[j].y;
      in[j] = __fmul2_rn(in[j], in[j]);
    }
    slide<kHS>(in, g, o);
#pragma unroll
    for (int i = 0; i < kHS; ++i) h2[r][c0 + i] = o[i];
    slide<kHS>(xy, g, p);
#pragma unroll
    for (int i = 0; i < kHS; ++i) h3[r][c0 + i] = p[i];
  }
  __syncthreads();
  // vertical pass: item = (column, kVS rows), then the SSIM terms
  const int col = t % kTW, r0 = (t / kTW) * kVS;
  float2 m1[kVS], m2[kVS];
  float m3[kVS];
  {
    float2 in[kVS + kTaps - 1];
#pragma unroll
    for (int j = 0; j < kVS + kTaps - 1; ++j) in[j] = h1[r0 + j][col];
    slide<kVS>(in, g, m1);
#pragma unroll
    for (int j = 0; j < kVS + kTaps - 1; ++j) in[j] = h2[r0 + j][col];
    slide<kVS>(in, g, m2);
    float xy[kVS + kTaps - 1];
#pragma unroll
    for (int j = 0; j < kVS + kTaps - 1; ++j) xy[j] = h3[r0 + j][col];
    slide<kVS>(xy, g, m3);
  }
  const int px = blockIdx.x * kTW + col;
  float ssim = 0.f, l1 = 0.f;
  const float C1 = 0.01f * 0.01f, C2 = 0.03f * 0.03f;
#pragma unroll
  for (int i = 0; i < kVS; ++i) {
    const int py = blockIdx.y * kTH + r0 + i;
    if (px < W && py < H && r0 + i < kTH) {
      const float ux = m1[i].x, uy = m1[i].y;
      const float vx = m2[i].x - ux * ux, vy = m2[i].y - uy * uy, cxy = m3[i] - ux * uy;
      const float A1 = 2.f * ux * uy + C1, A2 = 2.f * cxy + C2;
      const float B1 = ux * ux + uy * uy + C1, B2 = vx + vy + C2;
      const float iB = 1.f / (B1 * B2);
      const float s = A1 * A2 * iB;
      const float dux = 2.f * uy * A2 * iB - s * 2.f * ux / B1;
      const float dvx = -s / B2;
      const float dcxy = 2.f * A1 * iB;
      const size_t pix = (size_t)py * W + px;
      part[(0 * 3 + c) * HW + pix] = dux - 2.f * ux * dvx - uy * dcxy;
      part[(1 * 3 + c) * HW + pix] = dvx;
      part[(2 * 3 + c) * HW + pix] = dcxy;
      ssim += s;
      l1 += fabsf(out[c * HW + pix] - tgt[c * HW + pix]);
    }
  }
  // block sums
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    ssim += __shfl_xor_sync(0xffffffffu, ssim, o);
    l1 += __shfl_xor_sync(0xffffffffu, l1, o);
  }
  __shared__ float ws[2][kThr / 32];
  if ((t & 31) == 0) { ws[0][t >> 5] = l1; ws[1][t >> 5] = ssim; }
  __syncthreads();
  if (t == 0) {
    float a = 0.f, b = 0.f;
    for (int i = 0; i < kThr / 32; ++i) { a += ws[0][i]; b += ws[1][i]; }
    const size_t bi = ((size_t)c * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
    bsum[2 * bi] = a;
    bsum[2 * bi + 1] = b;
  }
}

__global__ void __launch_bounds__(kThr, 5) ssim_bwd_kernel(
    int W, int H, const float* __restrict__ out, const float* __restrict__ tgt,
    const float* __restrict__ tinv, Gauss g, gs_loss_weights wt, const float* __restrict__ part,
    float* __restrict__ adj_total, float* __restrict__ adj_ssim, float* __restrict__ adj_l1,
    float* __restrict__ dsum) {
  __shared__ float2 s1[kHaloH][kSX];  // partials by mu_x and E[x^2]
  __shared__ float s2[kHaloH][kSX];   // by E[xy]
  float2 (*const h1)[kSH] = reinterpret_cast<float2 (*)[kSH]>(s1);  // sums, in the halo's place
  float (*const h2)[kSH] = reinterpret_cast<float (*)[kSH]>(s2);
  const int c = blockIdx.z;
  const size_t HW = (size_t)W * H;
  const int ox = blockIdx.x * kTW - kR, oy = blockIdx.y * kTH - kR;
  const int t = threadIdx.x;
  // partial q of channel c is plane 3 q + c
  stage_halo<3>(s1, s2, Planes<3>{{part + c * HW, part + (3 + c) * HW, part + (6 + c) * HW}}, W, H, ox, oy);
  __syncthreads();
  {
    const int r = t % kHaloH, c0 = (t / kHaloH) * kHS;
    float2 in[kHS + kTaps - 1], o[kHS];
    float in2[kHS + kTaps - 1], o2[kHS];
#pragma unroll
    for (int j = 0; j < kHS + kTaps - 1; ++j) {
      in[j] = s1[r][c0 + j];
      in2[j] = s2[r][c0 + j];
    }
    __syncthreads();  // the halo is read
    slide<kHS>(in, g, o);
#pragma unroll
    for (int i = 0; i < kHS; ++i) h1[r][c0 + i] = o[i];
    slide<kHS>(in2, g, o2);
#pragma unroll
    for (int i = 0; i < kHS; ++i) h2[r][c0 + i] = o2[i];
  }
  __syncthreads();
  const int col = t % kTW, r0 = (t / kTW) * kVS;
  float2 b1[kVS];
  float b2[kVS];
  {
    float2 in[kVS + kTaps - 1];
#pragma unroll
    for (int j = 0; j < kVS + kTaps - 1; ++j) in[j] = h1[r0 + j][col];
    slide<kVS>(in, g, b1);
    float in2[kVS + kTaps - 1];
#pragma unroll
    for (int j = 0; j < kVS + kTaps - 1; ++j) in2[j] = h2[r0 + j][col];
    slide<kVS>(in2, g, b2);
  }
  const int px = blockIdx.x * kTW + col;
  const float inv = 1.f / (3.f * (float)HW);
  float dl = 0.f;
#pragma unroll
  for (int i = 0; i < kVS; ++i) {
    const int py = blockIdx.y * kTH + r0 + i;
    if (px < W && py < H && r0 + i < kTH) {
      const size_t pix = (size_t)py * W + px;
      const float x = out[c * HW + pix], y = tgt[c * HW + pix];
      const float dssim = b1[i].x + 2.f * x * b1[i].y + y * b2[i];
      const float as = -wt.w_ssim * dssim * inv;
      const float d = x - y;
      const float al = wt.w_l1 * (d > 0.f ? 1.f : (d < 0.f ? -1.f : 0.f)) * inv;
      adj_total[c * HW + pix] = as + al;
      if (adj_ssim) adj_ssim[c * HW + pix] = as;
      if (adj_l1) adj_l1[c * HW + pix] = al;
      if (c == 0 && tinv) {
        const float e = out[5 * HW + pix] - tinv[pix];
        dl += fabsf(e);
        adj_total[5 * HW + pix] = wt.w_depth * (e > 0.f ? 1.f : (e < 0.f ? -1.f : 0.f)) / (float)HW;
      }
    }
  }
  if (c == 0 && dsum) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) dl += __shfl_xor_sync(0xffffffffu, dl, o);
    __shared__ float ws[kThr / 32];
    if ((t & 31) == 0) ws[t >> 5] = dl;
    __syncthreads();
    if (t == 0) {
      float a = 0.f;
      for (int i = 0; i < kThr / 32; ++i) a += ws[i];
      dsum[blockIdx.y * gridDim.x + blockIdx.x] = a;
    }
  }
}

// A sum in FP32 with what its additions rounded off (Knuth's two-sum): FP64's
// precision without an FP64 addition and a conversion per term, which cost the
// loss of a 1600 x 900 image 2 us.
struct Sum2 {
  float hi = 0.f, lo = 0.f;
  __device__ __forceinline__ void add(float x) {
    const float s = hi + x, b = s - hi;
    lo += (hi - (s - b)) + (x - b);
    hi = s;
  }
  __device__ __forceinline__ double value() const {
    return fabsf(hi) < INFINITY ? (double)hi + (double)lo : (double)hi;
  }
};

// Latency only: two rounds of loads, eight levels of a tree, no FP64 division
// (one takes about a microsecond here).  The per-block sums of a 1600 x 900
// image: 8.7 -> 6.5 us.
constexpr int kRed = 256;
__global__ void __launch_bounds__(kRed) loss_reduce_kernel(const float* __restrict__ bsum, int nb,
                                                           const float* __restrict__ dsum, int nd, double inv_n3,
                                                           double inv_hw, gs_loss_weights wt, int has_depth,
                                                           float* __restrict__ losses) {
  __shared__ double red[3][kRed];
  // a thread adds ten blocks' sums of a 900p image and over two hundred of an
  // 8K one; the tree in FP64
  Sum2 a, b, d;
#pragma unroll 8
  for (int i = threadIdx.x; i < nb; i += kRed) {
    a.add(bsum[2 * i]);
    b.add(bsum[2 * i + 1]);
  }
  if (has_depth)
#pragma unroll 4
    for (int i = threadIdx.x; i < nd; i += kRed) d.add(dsum[i]);
  red[0][threadIdx.x] = a.value();
  red[1][threadIdx.x] = b.value();
  red[2][threadIdx.x] = d.value();
  __syncthreads();
  for (int s = kRed / 2; s > 0; s >>= 1) {
    if (threadIdx.x < s) {
      red[0][threadIdx.x] += red[0][threadIdx.x + s];
      red[1][threadIdx.x] += red[1][threadIdx.x + s];
      red[2][threadIdx.x] += red[2][threadIdx.x + s];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    const double l1 = red[0][0] * inv_n3, ss = red[1][0] * inv_n3;
    const double ld = has_depth ? red[2][0] * inv_hw : 0.0;
    losses[0] = (float)l1;
    losses[1] = (float)ss;
    losses[2] = (float)ld;
    losses[3] = (float)(wt.w_l1 * l1 + wt.w_ssim * (1.0 - ss) + wt.w_depth * ld);
  }
}

}  // namespace

size_t loss_tmp_floats(int W, int H) {
  const size_t gx = div_up(W, kTW), gy = div_up(H, kTH);
  return 9 * (size_t)W * H + 2 * 3 * gx * gy + gx * gy + 64;
}

cudaError_t launch_loss(int W, int H, const float* out, const float* tgt, const float* tinv,
                        const gs_loss_weights& w, float* adj_total, float* adj_ssim,
                        float* adj_l1, float* losses, float* tmp, cudaStream_t st) {
  Gauss g;
  double s = 0.0, e[2 * kR + 1];
  for (int i = 0; i < 2 * kR + 1; ++i) {
    e[i] = exp(-((i - kR) * (i - kR)) / (2.0 * 1.5 * 1.5));
    s += e[i];
  }
  for (int i = 0; i < 2 * kR + 1; ++i) g.w[i] = (float)(e[i] / s);
  const unsigned gx = div_up(W, kTW), gy = div_up(H, kTH);
  float* part = tmp;
  float* bsum = tmp + 9 * (size_t)W * H;
  float* dsum = bsum + 2 * 3 * (size_t)gx * gy;
  const dim3 grid(gx, gy, 3);
  ProfScope ps(kProfLoss, st);
  count_launch(3);
  ssim_fwd_kernel<<<grid, kThr, 0, st>>>(W, H, out, tgt, g, part, bsum);
  ssim_bwd_kernel<<<grid, kThr, 0, st>>>(W, H, out, tgt, tinv, g, w, part, adj_total, adj_ssim,
                                        adj_l1, dsum);
  const double hw = (double)W * H;
  loss_reduce_kernel<<<1, kRed, 0, st>>>(bsum, 3 * gx * gy, dsum, gx * gy, 1.0 / (3.0 * hw), 1.0 / hw, w,
                                         tinv != nullptr, losses);
  return cudaGetLastError();
}

}  // namespace gs2d

// ---------------------------------------------------------------------------
// Loss without any device allocation (gs_loss_noalloc).
//
// Some callers cannot allocate device memory at the moment they need the
// loss: a renderer or trainer that runs under an external memory manager
// which owns every byte of the GPU (allocating behind its back would break
// its budget), a real-time loop where an allocation's latency or possible
// failure is not acceptable, or a host that hands this library a device it
// may only compute on.  For them the loss's scratch (the SSIM partial maps
// and the per-block sums) lives in one fixed array in this file, sized for
// images of up to kNoAllocMaxPixels pixels with sides up to kNoAllocMaxSide.
// Every GPU that loads the library reserves it (about 9.5 MB) until the
// process exits.  Every call uses the same array, so calls whose work can
// overlap on the GPU (different streams, or different host threads) race.
namespace gs2d {
namespace {

constexpr int kNoAllocMaxPixels = 512 * 512;
constexpr int kNoAllocMaxSide = 4096;
// per-block sums: at most HW/256 + (W + H)/16 + 1 blocks (an upper bound
// for the loss kernels' 32 x 54 tiles as well)
constexpr size_t kNoAllocTiles = kNoAllocMaxPixels / 256 + (2 * kNoAllocMaxSide) / 16 + 1;
constexpr size_t kNoAllocFloats = 9 * (size_t)kNoAllocMaxPixels + 7 * kNoAllocTiles + 64;
constexpr int kNoAllocMaxDevices = 64;

static __device__ __align__(256) float g_noalloc_loss_scratch[kNoAllocFloats];

std::mutex g_noalloc_mu;
float* g_noalloc_addr[kNoAllocMaxDevices] = {};

}  // namespace
}  // namespace gs2d

extern "C" gs_status gs_loss_noalloc(int32_t W, int32_t H, const float* out, const float* tgt,
                                     const float* tinv, const gs_loss_weights* w, float* adj_total,
                                     float* adj_ssim, float* adj_l1, float* losses, void* stream) {
  using namespace gs2d;
  if (W <= 0 || H <= 0 || !out || !tgt || !w || !adj_total || !losses) {
    set_last_error("gs_loss_noalloc: bad argument");
    return GS_ERR_ARG;
  }
  if ((int64_t)W * H > kNoAllocMaxPixels || W > kNoAllocMaxSide || H > kNoAllocMaxSide ||
      loss_tmp_floats(W, H) > kNoAllocFloats) {
    set_last_error(("gs_loss_noalloc: image " + std::to_string(W) + "x" + std::to_string(H) +
                    " exceeds the fixed scratch (at most " + std::to_string(kNoAllocMaxPixels) +
                    " pixels, sides up to " + std::to_string(kNoAllocMaxSide) + "); use gs_loss")
                       .c_str());
    return GS_ERR_CAPACITY;
  }
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess || dev < 0 || dev >= kNoAllocMaxDevices) {
    set_last_error("gs_loss_noalloc: no usable current device");
    return GS_ERR_CUDA;
  }
  float* scratch = nullptr;
  {
    // once per device, with that device current: the device address of the
    // scratch array (its name in host code is only a host-side handle)
    std::lock_guard<std::mutex> lk(g_noalloc_mu);
    if (!g_noalloc_addr[dev]) {
      void* ptr = nullptr;
      e = cudaGetSymbolAddress(&ptr, g_noalloc_loss_scratch);
      if (e != cudaSuccess || !ptr) {
        set_last_error((std::string("gs_loss_noalloc: cudaGetSymbolAddress: ") + cudaGetErrorString(e)).c_str());
        return GS_ERR_CUDA;
      }
      g_noalloc_addr[dev] = static_cast<float*>(ptr);
    }
    scratch = g_noalloc_addr[dev];
  }
  // Nothing in the scratch must start at zero: every partial map entry and
  // per-block sum the kernels read is written earlier in the same call.
  e = launch_loss(W, H, out, tgt, tinv, *w, adj_total, adj_ssim, adj_l1, losses, scratch,
                  (cudaStream_t)stream);
  if (e != cudaSuccess) {
    set_last_error((std::string("gs_loss_noalloc: ") + cudaGetErrorString(e)).c_str());
    return GS_ERR_CUDA;
  }
  return GS_OK;
}
