// Visible frequency of points over many views (Sec. 4, crop volume
// estimation): each ground-truth point is an isotropic 3D Gaussian of
// standard deviation sigma, and its count is the number of views in which
// the rasterizer would keep it: in front of the near plane, with the
// 3-sigma square of its EWA-projected footprint (sigma^2 J J^T plus a low-pass
// of `lowpass` px^2, J the Jacobian of the perspective projection)
// overlapping the image.  Occlusion plays no part (the rasterizer's
// per-primitive visible mask).
//
// Two points per thread on the packed FP32 instructions, the views staged
// through shared memory in chunks; no memory traffic beyond the point itself,
// so the count over N points and V views is bound by instruction issue.  The
// definition costs about 90 instructions per (point, view) in front of the
// camera, most of them an IEEE division and two IEEE square roots.  Nearly
// every decision is clear without them, from comparisons that are linear in
// the point: a centre inside the image counts whatever its footprint, one
// further outside than a bound on its half-width does not.  The pairs left
// over, a few percent around the image's edge, are listed per thread and
// decided by the definition itself, many at a time (decided at once, they
// would hold up nearly every warp).  So the counts are the definition's.
// 8M points x 300 views: 5970 us by the definition alone, 4860 and 4720 us with
// finer tests and the rest decided at once, 2700 us so.
// The kept points' height range is a block reduction.
#include <math.h>

#include "gs2d_internal.cuh"

namespace gs2d {
namespace {

constexpr int kThreads = 256;
constexpr int kChunk = 128;  // views per shared-memory chunk
constexpr int kStep = 8;     // views between looks at the lists
constexpr int kList = 4 * kStep;

// What the clear-cut tests need of a view.  With (px, py, pz) the point in view
// space, X = fx px + (cx - W/2) pz and Y likewise are affine in the point:
// the projected centre's offset from the image centre times pz.
//   inside:  |X| < W/2 pz - t and |Y| < H/2 pz - t
//   outside: pz > z0 and (|X| > (W/2 + B) pz + A + t or |Y| > (H/2 + B) pz + A + t)
// A / pz + B bounds the half-width r of a footprint whose centre is at most
// Gm outside the image: 9 times the trace of its covariance is
//   9 sigma^2 / pz^2 (fx^2 + fy^2 + vx^2 + vy^2) + 18 lowpass,
// with |vx| = |X / pz - (cx - W/2)| <= W/2 + Gm + |cx - W/2|, and the root of
// a sum is at most the sum of the roots.  z0 is where A / pz + B = Gm; further
// outside by D, r grows by at most 3 sqrt(2) sigma / pz D, less than D beyond
// z0 >= 4.3 sigma.
// t = ku (|x| + |y| + |z|) + k0 covers the rounding of X and Y here and of the
// centre in the definition: each is a few operations on terms no larger than
// t's, so their errors are a few 2^-24 of those, and t takes 32 x 2^-24.
struct VisView {
  float4 a, b, c;  // X, Y and pz as affine functions of the point
  float4 d;        // W/2, H/2, ku, k0
  float4 e;        // W/2 + B, H/2 + B, A, z0
};

// One view's decision by the definition, for a point in front of it.
__device__ __forceinline__ bool vis_exact(const VisCam& k, float x, float y, float z, float pz, float sigma2,
                                       float lowpass) {
  const float px = fmaf(k.R[0], x, fmaf(k.R[1], y, fmaf(k.R[2], z, k.t[0])));
  const float py = fmaf(k.R[3], x, fmaf(k.R[4], y, fmaf(k.R[5], z, k.t[1])));
  const float iz = 1.f / pz;
  const float ux = px * iz, uy = py * iz;  // x/z, y/z
  const float gx = k.fx * iz, gy = k.fy * iz;
  // sigma^2 J J^T with J = [[gx, 0, -gx ux], [0, gy, -gy uy]]
  const float sxx = fmaf(sigma2 * gx * gx, fmaf(ux, ux, 1.f), lowpass);
  const float syy = fmaf(sigma2 * gy * gy, fmaf(uy, uy, 1.f), lowpass);
  const float sxy = sigma2 * gx * gy * ux * uy;
  const float mid = 0.5f * (sxx + syy), half = 0.5f * (sxx - syy);
  const float r = 3.f * sqrtf(mid + sqrtf(fmaf(half, half, sxy * sxy)));
  const float cx = fmaf(k.fx, ux, k.cx), cy = fmaf(k.fy, uy, k.cy);
  return cx + r > 0.f && cx - r < k.W && cy + r > 0.f && cy - r < k.H;
}

__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 both(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 affine(const float4& a, float2 x, float2 y, float2 z) {
  return fma2(both(a.x), x, fma2(both(a.y), y, fma2(both(a.z), z, both(a.w))));
}

__global__ void __launch_bounds__(kThreads) vis_count_kernel(const float* __restrict__ pts, int64_t n,
                                                             float sigma2, float lowpass, float near_plane,
                                                             const VisCam* __restrict__ cams,
                                                             const VisView* __restrict__ views, int nviews,
                                                             uint32_t* __restrict__ counts) {
  __shared__ VisCam sc[kChunk];
  __shared__ VisView sv[kChunk];
  __shared__ uint16_t list[kList][kThreads];  // open pairs of a thread: view, second point << 8
  const int64_t j0 = (int64_t)blockIdx.x * (2 * kThreads) + threadIdx.x, j1 = j0 + kThreads;
  const bool live0 = j0 < n, live1 = j1 < n;
  const float2 x = make_float2(live0 ? pts[3 * j0] : 0.f, live1 ? pts[3 * j1] : 0.f);
  const float2 y = make_float2(live0 ? pts[3 * j0 + 1] : 0.f, live1 ? pts[3 * j1 + 1] : 0.f);
  const float2 z = make_float2(live0 ? pts[3 * j0 + 2] : 0.f, live1 ? pts[3 * j1 + 2] : 0.f);
  // (a point out of the ordinary gets an infinite t, as such a view does)
  float2 m = make_float2(fabsf(x.x) + fabsf(y.x) + fabsf(z.x), fabsf(x.y) + fabsf(y.y) + fabsf(z.y));
  if (!(m.x < 1e15f)) m.x = INFINITY;
  if (!(m.y < 1e15f)) m.y = INFINITY;
  uint32_t c0 = 0u, c1 = 0u;
  int open = 0;  // entries of this thread's list
  const int per = (nviews + (int)gridDim.y - 1) / (int)gridDim.y;
  const int vend = min(nviews, per * ((int)blockIdx.y + 1));
  for (int v0 = per * (int)blockIdx.y; v0 < vend; v0 += kChunk) {
    const int nv = min(kChunk, vend - v0);
    __syncthreads();
    for (int i = threadIdx.x; i < nv; i += kThreads) {
      sc[i] = cams[v0 + i];
      sv[i] = views[v0 + i];
    }
    __syncthreads();
    for (int i0 = 0; i0 < nv; i0 += kStep) {
      const int i1 = min(i0 + kStep, nv);
      for (int i = i0; i < i1; ++i) {
        const VisView& v = sv[i];
        const float2 pz = affine(v.c, x, y, z);  // the definition's, bit for bit
        const float2 X = affine(v.a, x, y, z), Y = affine(v.b, x, y, z);
        const float2 t = fma2(both(v.d.z), m, both(v.d.w)), u = make_float2(-t.x, -t.y), s = add2(t, both(v.e.z));
        const float2 bx = fma2(both(v.d.x), pz, u), by = fma2(both(v.d.y), pz, u);
        const float2 ox = fma2(both(v.e.x), pz, s), oy = fma2(both(v.e.y), pz, s);
        const bool in0 = fabsf(X.x) < bx.x && fabsf(Y.x) < by.x, in1 = fabsf(X.y) < bx.y && fabsf(Y.y) < by.y;
        const bool out0 = pz.x > v.e.w && (fabsf(X.x) > ox.x || fabsf(Y.x) > oy.x);
        const bool out1 = pz.y > v.e.w && (fabsf(X.y) > ox.y || fabsf(Y.y) > oy.y);
        if (pz.x > near_plane) {
          c0 += in0 ? 1u : 0u;
          if (!in0 && !out0) list[open++][threadIdx.x] = (uint16_t)i;
        }
        if (pz.y > near_plane) {
          c1 += in1 ? 1u : 0u;
          if (!in1 && !out1) list[open++][threadIdx.x] = (uint16_t)(i | 256);
        }
      }
      // the next step may add two entries per view
      const int longest = __reduce_max_sync(0xffffffffu, open);
      if (longest <= kList - 2 * kStep && i1 < nv) continue;
      for (int e = 0; e < longest; ++e) {
        if (e >= open) continue;
        const int w = list[e][threadIdx.x], i = w & 255;
        const bool second = (w & 256) != 0;
        const float qx = second ? x.y : x.x, qy = second ? y.y : y.x, qz = second ? z.y : z.x;
        const VisCam& k = sc[i];
        const float pz = fmaf(k.R[6], qx, fmaf(k.R[7], qy, fmaf(k.R[8], qz, k.t[2])));
        const uint32_t one = vis_exact(k, qx, qy, qz, pz, sigma2, lowpass) ? 1u : 0u;
        c0 += second ? 0u : one;
        c1 += second ? one : 0u;
      }
      open = 0;
    }
  }
  if (gridDim.y == 1) {
    if (live0) counts[j0] += c0;
    if (live1) counts[j1] += c1;
  } else {
    if (live0 && c0 != 0u) atomicAdd(&counts[j0], c0);
    if (live1 && c1 != 0u) atomicAdd(&counts[j1], c1);
  }
}

// The views' affine forms, computed in double from the cameras (one thread per view).
// A view out of the ordinary gets an infinite t, with which neither clear-cut
// test ever holds: the ranges below keep everything the tests and the
// definition compute finite, or let it overflow in a way the tests allow for.
__global__ void vis_views_kernel(const VisCam* __restrict__ cams, int nviews, float sigma, float lowpass,
                                 bool fast, VisView* __restrict__ views) {
  const int v = blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= nviews) return;
  const VisCam k = cams[v];
  const double hx = (double)k.cx - 0.5 * (double)k.W, hy = (double)k.cy - 0.5 * (double)k.H;
  float a[4], b[4];
  for (int i = 0; i < 4; ++i) {
    const double r0 = i < 3 ? k.R[i] : k.t[0], r1 = i < 3 ? k.R[3 + i] : k.t[1], r2 = i < 3 ? k.R[6 + i] : k.t[2];
    a[i] = (float)((double)k.fx * r0 + hx * r2);
    b[i] = (float)((double)k.fy * r1 + hy * r2);
  }
  float rmax = 1.f;
  for (int i = 0; i < 9; ++i) rmax = fmaxf(rmax, fabsf(k.R[i]));
  const float tmax = fmaxf(fmaxf(fabsf(k.t[0]), fabsf(k.t[1])), fabsf(k.t[2]));
  const float scale = fmaxf(k.fx, k.fy) + (float)(fabs(hx) + fabs(hy)) + k.W + k.H;
  const float u = 32.f * 5.9604645e-8f;
  bool plain = fast && fminf(k.fx, k.fy) > 1e-3f && scale < 1e6f && rmax < 4.f && tmax < 1e15f;
  for (int i = 0; i < 9; ++i) plain = plain && k.R[i] == k.R[i];
  for (int i = 0; i < 3; ++i) plain = plain && k.t[i] == k.t[i];
  VisView o;
  o.a = make_float4(a[0], a[1], a[2], a[3]);
  o.b = make_float4(b[0], b[1], b[2], b[3]);
  o.c = make_float4(k.R[6], k.R[7], k.R[8], k.t[2]);
  o.d = make_float4(0.5f * k.W, 0.5f * k.H, plain ? u * scale * rmax : 0.f, plain ? u * scale * tmax : INFINITY);
  const double B = 3.003 * sqrt(2.0 * (double)lowpass), Gm = 0.125 * ((double)k.W + (double)k.H) + 4.0 * B + 16.0;
  const double vx = 0.5 * (double)k.W + Gm + fabs(hx), vy = 0.5 * (double)k.H + Gm + fabs(hy);
  const double A = 3.003 * (double)sigma * sqrt((double)k.fx * k.fx + (double)k.fy * k.fy + vx * vx + vy * vy);
  o.e = make_float4(0.5f * k.W + (float)B, 0.5f * k.H + (float)B, (float)A,
                    fmaxf((float)(1.001 * A / (Gm - B)), 4.3f * sigma));
  views[v] = o;
}

// Points seen in at least min_count views: keep mask, and the lowest and
// highest world z among them (ordered-int atomics on the float bits).
__device__ __forceinline__ int ord(float f) {
  const int b = __float_as_int(f);
  return b >= 0 ? b : b ^ 0x7FFFFFFF;
}
__device__ __forceinline__ float unord(int b) { return __int_as_float(b >= 0 ? b : b ^ 0x7FFFFFFF); }

__global__ void vis_init_kernel(int* __restrict__ zr) {
  zr[0] = 0x7FFFFFFF;         // min (as an ordered int)
  zr[1] = (int)0x80000000;    // max
}

__global__ void __launch_bounds__(kThreads) vis_keep_kernel(const float* __restrict__ pts, int64_t n,
                                                            const uint32_t* __restrict__ counts, uint32_t min_count,
                                                            uint8_t* __restrict__ keep, int* __restrict__ zr) {
  int lo = 0x7FFFFFFF, hi = (int)0x80000000;
  for (int64_t j = (int64_t)blockIdx.x * kThreads + threadIdx.x; j < n; j += (int64_t)gridDim.x * kThreads) {
    const bool k = counts[j] >= min_count;
    keep[j] = k ? 1u : 0u;
    if (k) {
      const int o = ord(pts[3 * j + 2]);
      lo = min(lo, o);
      hi = max(hi, o);
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    lo = min(lo, __shfl_xor_sync(0xffffffffu, lo, o));
    hi = max(hi, __shfl_xor_sync(0xffffffffu, hi, o));
  }
  if ((threadIdx.x & 31) == 0) {
    atomicMin(&zr[0], lo);
    atomicMax(&zr[1], hi);
  }
}

__global__ void vis_range_kernel(const int* __restrict__ zr, float* __restrict__ zrange) {
  const bool any = zr[0] != 0x7FFFFFFF;
  zrange[0] = any ? unord(zr[0]) : NAN;
  zrange[1] = any ? unord(zr[1]) : NAN;
}

}  // namespace

size_t visibility_tmp_bytes(int nviews) { return sizeof(VisView) * (size_t)nviews; }

cudaError_t launch_visibility_count(const float* pts, int64_t n, float sigma, float lowpass, float near_plane,
                                    const VisCam* cams, int nviews, void* tmp, uint32_t* counts, cudaStream_t st) {
  if (n <= 0 || nviews <= 0) return cudaSuccess;
  ProfScope ps(kProfContrib, st);
  count_launch(2);
  VisView* views = static_cast<VisView*>(tmp);
  // the clear-cut tests suppose a point in front of the camera and a footprint
  // of finite size; other settings take the definition throughout
  const bool fast = near_plane > 1e-3f && sigma < 1e6f && lowpass < 1e6f;
  vis_views_kernel<<<div_up(nviews, 64), 64, 0, st>>>(cams, nviews, sigma, lowpass, fast, views);
  // Points that fill the GPU twice over keep their views together; fewer share
  // them out, 16 views or more to a block (a launch's length is then some 16
  // views, not all of them).  300 views, shared out / together, us: 10k points
  // 24 / 75, 100k 59 / 88, 300k 128 / 141, 600k 237 / 244, 1M 374 / 376.
  const unsigned blocks = div_up(n, 2 * kThreads), want = 8u * sm_count();
  const unsigned most = (unsigned)((nviews + 15) / 16);
  unsigned split = blocks >= want ? 1u : (want + blocks - 1) / blocks;
  if (split > most) split = most;
  vis_count_kernel<<<dim3(blocks, split), kThreads, 0, st>>>(pts, n, sigma * sigma, lowpass, near_plane, cams, views,
                                                             nviews, counts);
  return cudaGetLastError();
}

cudaError_t launch_visibility_keep(const float* pts, int64_t n, const uint32_t* counts, uint32_t min_count,
                                   uint8_t* keep, float* zrange, int* tmp, cudaStream_t st) {
  ProfScope ps(kProfContrib, st);
  count_launch(3);
  vis_init_kernel<<<1, 1, 0, st>>>(tmp);
  if (n > 0) {
    const unsigned g = div_up(n, kThreads) < 1216u ? div_up(n, kThreads) : 1216u;
    vis_keep_kernel<<<g, kThreads, 0, st>>>(pts, n, counts, min_count, keep, tmp);
  }
  vis_range_kernel<<<1, 1, 0, st>>>(tmp, zrange);
  return cudaGetLastError();
}

}  // namespace gs2d
