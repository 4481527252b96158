// Per-pixel compositing (forward) and its adjoint (reverse replay).
//
// Forward (Eq. 1, Sec. 3.1, with the 2DGS surfel model and the low-pass
// filter of Sec. 3.2): one CTA of 128 threads per 16 x 16 tile; each lane
// group of eight covers a 4 x 4 block of pixels and each thread two pixels of
// one column, two rows apart, so that an entry read from shared memory serves
// two pixels and the two per-pixel dependency chains interleave.  The tile's
// depth-sorted surfel list is staged through shared memory in batches of
// 256 entries; each group walks the entries whose footprint can touch its
// block (the block masks that launch_ranges made, turned into one index list
// per group and batch), so the four groups of a warp evaluate four entries
// side by side.  Each pixel intersects its ray with the surfel plane
// (rho_obj), takes the screen-space filter (rho_scr) where smaller, and
// composites front to back until the transmittance would drop below T_min.
//
// Backward: the same tiles replay each pixel's list back to front from the
// final transmittance, T_before = T_after / (1 - alpha), with suffix sums
// for d L / d alpha.  Each warp stages and walks its own window on the list,
// without barriers of the CTA.  A thread adds the gradients of its two pixels,
// the group reduces them with a reduce-scatter of shuffles (one reduction per
// four entries and 16 pixels each) and adds its sums to the surfel's gradient
// row in global memory, in double: in float the order of the many small
// additions doubled the gradients' error.
//
// Both are bound by instruction issue, so the time is (group, entry) steps
// times instructions per step.  With one list per warp (8 x 8 pixels) only 10
// (4M-surfel orbit view) to 18 (1M aerial view) of a step's 32 lanes blended
// anything; 4 x 4 blocks cost a warp the longest of its four lists instead of
// their union, and packed FP32 does a thread's two pixels in one instruction.
// Measured, us (1M-surfel 1600 x 900 view forward and backward, 4M-surfel
// 1080p view forward, the four backwards of a 4M-surfel training step):
//   one list per warp, scalar FP32          501  1160  1148  9640
//   one list per group                      335   980   690  7400
//   packed FP32                             294   912   583  6550
//   backward without CTA barriers           296   768   583  5390
#include <math.h>

#include "gs2d_internal.cuh"

namespace gs2d {
namespace {

constexpr int kThreads = 128;  // threads per tile CTA, two pixels each
constexpr int kBatch = 256;    // list entries staged per batch
constexpr int kTilePix = 2 * kThreads;  // pixels of a tile, two per thread

// Hardware approximations (relative error about 2^-22), the same
// instructions in both blends so that the replay reproduces the forward's
// decisions exactly.
__device__ __forceinline__ float rcp_approx(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float ex2_approx(float x) {
  float r;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
// Packed FP32 pairs: one instruction does the same rounded operation on both
// halves; a scalar operand spread over both (bc) and a negated one cost
// nothing.  Measured on this GPU: 1.87 packed against 2.6 scalar FMAs per SM
// and clock, so a pair of pixels takes half the issue slots and 0.7 of the
// FMA pipe's time.  Selects and compares run at 1.9 per SM and clock, as
// dear as a packed FMA: the code below keeps them few.
__device__ __forceinline__ float2 bc(float x) { return make_float2(x, x); }
__device__ __forceinline__ float2 neg2(float2 x) { return make_float2(-x.x, -x.y); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 rcp2(float2 x) { return make_float2(rcp_approx(x.x), rcp_approx(x.y)); }
__device__ __forceinline__ float2 sel2(bool a, bool b, float2 x, float2 y) {
  return make_float2(a ? x.x : y.x, b ? x.y : y.y);
}
constexpr float kNegHalfLog2e = -0.72134752044448170f;  // -log2(e) / 2

// Pixels of thread t within its tile: warp w covers columns 8 (w & 1) .. +7
// and rows 8 (w >> 1) .. +7, its lane group g = (l >> 3) the 4 x 4 block at
// column 4 (g & 1), row 4 (g >> 1) of those, and lane l column l & 3 and rows
// (l >> 2) & 1 and that + kRowStep of the group's block.
constexpr int kRowStep = 2;  // rows between a thread's two pixels
__device__ __forceinline__ int local_x(int t) { return (((t >> 5) & 1) << 3) | (((t >> 3) & 1) << 2) | (t & 3); }
__device__ __forceinline__ int local_y(int t) { return ((t >> 6) << 3) | (((t >> 4) & 1) << 2) | ((t >> 2) & 1); }

// Staged entry: s0 = (-c.x, -c.y relative to the tile origin, e.x, e.y),
// s1 = Jh, s2 = (p_z, opacity, r, g), s3 = (b, n.x, n.y, n.z), s4 = Jl,
// s5 = (nu0h, nv0h, nu0l, nv0l).
//
// Tile-relative ray-splat coordinates.  For a pixel at offset (lx, ly) from
// the tile origin o, Ji d = Ji (o - c) + Ji (lx, ly) = n0 + Ji (lx, ly).  Held
// in FP32 as Ji d, the coordinates of an ill-conditioned footprint (a nearly
// edge-on or elongated disk: large Ji, pixel far from c along the long axis)
// would carry an absolute error of about 2^-24 |Ji| |d|, far above the
// error of the exact value near the support boundary.  The preprocess splits
// Ji = Jh + Jl and the offset of the surfel's first tile origin o_ref,
// Ji (o_ref - c) = nref_h + nref_l, on a power-of-two grid 2^g chosen from the
// magnitudes over the surfel's tile rectangle: the high parts (nref_h on
// multiples of 2^g, Jh on multiples of 2^(g+1)) are so coarse that
// nref_h + Jh (o - o_ref) + Jh (lx, ly) is exact in FP32 (o - o_ref are
// multiples of 16, lx, ly half-integers below 16, every partial sum stays
// below 2^(g+24)); the low parts (about 2^g) carry the rest with negligible
// FP32 rounding.  Per (entry, tile) the staging forms
// n0h = nref_h + Jh (o - o_ref) (exact) and n0l = nref_l + Jl (o - o_ref) with
// four FMAs each; per pixel
// Ji d = [n0h + Jh (lx, ly)] + [n0l + Jl (lx, ly)] is then accurate to the
// FP32 rounding of the result itself, whatever the conditioning of Ji.
struct Staged {
  float4 s0, s1, s2, s3, s4, s5;
};

__device__ __forceinline__ Staged stage_entry(const float4* __restrict__ rec, uint32_t s, int tx0, int ty0) {
  const float4* R = rec + (size_t)s * kRecF4;
  const float4 r0 = R[0], r1 = R[1], r2 = R[2], r3 = R[3], r4 = R[4], r5 = R[5], r6 = R[6];
  Staged e;
  // centre relative to the tile origin: (c_hi - x0) + c_lo keeps the
  // offset accurate to its own rounding
  e.s0 = make_float4(-__fadd_rn(__fsub_rn(r0.x, (float)tx0), r0.z),
                     -__fadd_rn(__fsub_rn(r0.y, (float)ty0), r0.w), r2.x, r2.y);
  e.s2 = make_float4(r2.z, r2.w, r3.x, r3.y);
  e.s3 = make_float4(r3.z, r3.w, r4.x, r4.y);
  e.s1 = r1;
  e.s4 = r5;
  // n0 at this tile's origin (o - o_ref: multiples of 16, exact); the low
  // part's grid rounding q moves to the high part (both sums exact), so the
  // low part stays below 2^(g-1) whatever the tile's distance from o_ref
  const uint32_t rt = __float_as_uint(r6.z);
  const float dox = (float)(tx0 - (int)(rt & 0xFFFFu) * kTile), doy = (float)(ty0 - (int)(rt >> 16) * kTile);
  const float ug = r6.w, dg = __frcp_rn(ug);
  const float hu = __fmaf_rn(r1.x, dox, __fmaf_rn(r1.y, doy, r4.z));
  const float hv = __fmaf_rn(r1.z, dox, __fmaf_rn(r1.w, doy, r4.w));
  const float lu = __fmaf_rn(r5.x, dox, __fmaf_rn(r5.y, doy, r6.x));
  const float lv = __fmaf_rn(r5.z, dox, __fmaf_rn(r5.w, doy, r6.y));
  const float qu = __fmul_rn(rintf(__fmul_rn(lu, ug)), dg), qv = __fmul_rn(rintf(__fmul_rn(lv, ug)), dg);
  e.s5 = make_float4(__fadd_rn(hu, qu), __fadd_rn(hv, qv), __fsub_rn(lu, qu), __fsub_rn(lv, qv));
  return e;
}

// Per lane group of eight, the batch's entries whose footprint may reach the
// group's 4 x 4 pixel block, as a list of indices into the batch: the four
// groups of a warp walk their own lists side by side, so an entry costs a
// group nothing where it misses the group's block.
// sm holds the entries' block masks (bit 4 w + g); entry e is listed for a
// group only below the group's limit.  Returns the length of the caller's
// group's list.
template <int NB>
constexpr int kListStride = NB + 4;  // padded: a walk reads one index past its list
template <int NB>
__device__ __forceinline__ int group_lists(const uint16_t* sm, int nb, int warp, int lane,
                                           uint8_t (*list)[kListStride<NB>], int limit = NB) {
  const uint32_t lt = (1u << lane) - 1u;
  int base[4] = {0, 0, 0, 0}, lim[4];
#pragma unroll
  for (int g = 0; g < 4; ++g) lim[g] = min(__shfl_sync(0xffffffffu, limit, 8 * g), nb);
#pragma unroll
  for (int j = 0; j < NB / 32; ++j) {
    const int e = 32 * j + lane;
    const uint32_t m = e < nb ? (uint32_t)sm[e] >> (4 * warp) : 0u;
#pragma unroll
    for (int g = 0; g < 4; ++g) {
      const bool in = ((m >> g) & 1u) && e < lim[g];
      const uint32_t b = __ballot_sync(0xffffffffu, in);
      if (in) list[g][base[g] + __popc(b & lt)] = (uint8_t)e;
      base[g] += __popc(b);
    }
  }
  __syncwarp();
  const int g = lane >> 3;
  return g == 0 ? base[0] : (g == 1 ? base[1] : (g == 2 ? base[2] : base[3]));
}

// One warp's window on its tile's list: the entries that reach its 8 x 8
// block, staged 32 at a time into the two halves of a ring, and for each of
// the warp's four lane groups the ring slots of the entries that reach the
// group's 4 x 4 block, in walking order.
constexpr int kHalf = 32;
constexpr int kRing = 2 * kHalf;
constexpr int kQueue = kRing;
constexpr int kNoMore = 1 << 30;
struct WarpSmem {
  // slot kRing: an entry that no pixel is near, for the groups whose list is used up
  float4 s0[kRing + 1], s1[kRing + 1], s2[kRing + 1], s3[kRing + 1], s4[kRing + 1], s5[kRing + 1];
  uint2 meta[kRing + 1];   // list position, surfel
  uint2 q[kQueue];         // entries found but not yet staged (a ring): position, surfel
  uint8_t qm[kQueue];      // and their group masks
  uint16_t list[4][kRing];  // per group, byte offsets of ring slots (16 x slot; a ring of its own)
};

// Walks list positions [p0, p1) of a tile (front to back, or back to front
// when kBack) for one warp.  body(k, i) is called with every lane: k is the
// offset (16 x ring slot) of the lane's group's next entry and i the number
// of entries of its list walked so far, this one included; a group whose list
// is used up for now gets an entry that misses every pixel.  A lane that needs
// no more entries sets i to kNoMore (or starts with it).  kBack: the group
// takes only entries below its limit.  Returns the lane's i.
//
// The warps of a CTA share no data and no barrier: with one staging per CTA
// and batch, a quarter of the warps' time went to waiting for the slowest
// warp and for the staging loads.  A group may run ahead of the others by
// up to one half of the ring, which evens out most of the difference between
// the groups' lists (the older half is refilled when all groups are past it).
// Element of a staged array at a byte offset that is 16 times its slot.
__device__ __forceinline__ float4 at16(const float4* a, int k) {
  return *reinterpret_cast<const float4*>(reinterpret_cast<const char*>(a) + k);
}
__device__ __forceinline__ uint2 at16(const uint2* a, int k) {
  return *reinterpret_cast<const uint2*>(reinterpret_cast<const char*>(a) + k / 2);
}

template <bool kBack, class Body>
__device__ __forceinline__ int walk_list(WarpSmem& sm, const float4* __restrict__ rec,
                                         const uint16_t* __restrict__ masks, const uint32_t* __restrict__ vals, int p0,
                                         int p1, int limit, int tx0, int ty0, int blk, int i, Body body) {
  constexpr unsigned kFull = 0xffffffffu;
  const int lane = threadIdx.x & 31, g = lane >> 3;
  const uint32_t lt = (1u << lane) - 1u;
  int scan = kBack ? p1 : p0, qn = 0, q0 = 0;
  uint32_t pm = 0u, pv = 0u;  // the next 32 entries' masks and surfels, loaded ahead
  auto left = [&] { return kBack ? scan > p0 : scan < p1; };
  auto at = [&] { return kBack ? scan - 1 - lane : scan + lane; };
  auto load = [&] {
    const int e = at();
    const bool in = kBack ? e >= p0 : e < p1;
    pm = in ? masks[e] : 0u;
    pv = in ? vals[e] : 0u;
  };
  load();
  if (lane == 0) {
    sm.s0[kRing] = make_float4(1e15f, 1e15f, 0.f, 0.f);
    sm.s1[kRing] = sm.s3[kRing] = sm.s4[kRing] = make_float4(0.f, 0.f, 0.f, 0.f);
    sm.s2[kRing] = make_float4(1.f, 0.f, 0.f, 0.f);
    sm.s5[kRing] = make_float4(__int_as_float(0x7fffffff), 0.f, 0.f, 0.f);
    sm.meta[kRing] = make_uint2(0x7fffffffu, 0u);
  }
  // entries staged so far for the lane's group, and for all four groups modulo
  // the ring (one byte each); mid: those of the older half
  int end = 0, h = 0;
  uint32_t cnt = 0u;
  for (;;) {
    int mid = end;
    const bool fill = qn > 0 || left();
    if (fill) {
      __syncwarp();  // every lane is done with the older half
      while (qn < kHalf && left()) {
        const int e = at();
        uint32_t m = (pm >> (4 * blk)) & 15u;
        const uint32_t v = pv;
        if constexpr (kBack) {
#pragma unroll
          for (int j = 0; j < 4; ++j)
            if (e >= __shfl_sync(kFull, limit, 8 * j)) m &= ~(1u << j);
        }
        scan += kBack ? -32 : 32;
        if (left()) load();
        const uint32_t b = __ballot_sync(kFull, m != 0u);
        if (m != 0u) {
          const int slot = (q0 + qn + __popc(b & lt)) & (kQueue - 1);
          sm.q[slot] = make_uint2((uint32_t)e, v);
          sm.qm[slot] = (uint8_t)m;
        }
        qn += __popc(b);
      }
      __syncwarp();
      const int nb = min(qn, kHalf);
      const int slot = h * kHalf + lane;
      uint32_t m = 0u;
      if (lane < nb) {
        const uint2 x = sm.q[(q0 + lane) & (kQueue - 1)];
        m = sm.qm[(q0 + lane) & (kQueue - 1)];
        const Staged e = stage_entry(rec, x.y, tx0, ty0);
        sm.s0[slot] = e.s0;
        sm.s1[slot] = e.s1;
        sm.s2[slot] = e.s2;
        sm.s3[slot] = e.s3;
        sm.s4[slot] = e.s4;
        sm.s5[slot] = e.s5;
        sm.meta[slot] = make_uint2(x.x, x.y);
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const bool in = (m >> j) & 1u;
        const uint32_t b = __ballot_sync(kFull, in);
        if (in) sm.list[j][((cnt >> (8 * j)) + __popc(b & lt)) & (kRing - 1)] = (uint16_t)(16 * slot);
        cnt += (uint32_t)__popc(b) << (8 * j);
        end += g == j ? __popc(b) : 0;
      }
      cnt &= 0x3f3f3f3fu;
      qn -= nb;
      q0 += nb;
      __syncwarp();
      h ^= 1;
    } else {
      mid = end;
    }
    while (__any_sync(kFull, i < mid)) {
      int k = 16 * kRing;
      if (i < end) {
        k = sm.list[g][i & (kRing - 1)];
        ++i;
      }
      body(k, i);
    }
    if (!__any_sync(kFull, i < (fill ? kNoMore : end))) break;
  }
  return i;
}

// One entry against a thread's two pixels A and B (one column, kRowStep rows
// apart); the halves of each pair are the two pixels.
struct Pair {
  float dx;        // pixel offset from the projected centre (the column is shared)
  float2 dy;
  float2 nu, nv;   // Ji d
  float2 rden;     // 1 / (1 + e.d)
  float2 rho;      // min(rho_obj, rho_scr)
  float2 alpha;    // min(alpha_max, o exp(-rho / 2))
  bool objA, objB; // object-space branch
  bool hitA, hitB; // rho <= rho_max and alpha >= alpha_min
};

// The exact grid sums nu0h + Jh (lx, ly) plus the small low-part corrections
// (see Staged), then the ray-splat distance, the screen filter and alpha.
// Shared by every blend; explicit round-to-nearest operations so that
// the forward and the backward take bit-identical decisions.
__device__ __forceinline__ Pair eval_pair(float lx, float2 ly, float4 s0, float4 jh, float4 jl, float4 n0, float opac,
                                          const SetDev& set) {
  Pair q;
  const float su = __fmaf_rn(jh.x, lx, n0.x), sv = __fmaf_rn(jh.z, lx, n0.y);  // exact, the column's part
  const float cu = __fmaf_rn(jl.x, lx, n0.z), cv = __fmaf_rn(jl.z, lx, n0.w);
  q.nu = add2(fma2(bc(jh.y), ly, bc(su)), fma2(bc(jl.y), ly, bc(cu)));
  q.nv = add2(fma2(bc(jh.w), ly, bc(sv)), fma2(bc(jl.w), ly, bc(cv)));
  q.dx = __fadd_rn(lx, s0.x);
  q.dy = add2(ly, bc(s0.y));
  const float2 den = fma2(bc(s0.z), bc(q.dx), fma2(bc(s0.w), q.dy, bc(1.0f)));
  q.rden = rcp2(den);
  const float2 u = mul2(q.nu, q.rden), v = mul2(q.nv, q.rden);
  const float2 ro = fma2(u, u, mul2(v, v));
  const float2 rs = mul2(bc(set.sinv), fma2(bc(q.dx), bc(q.dx), mul2(q.dy, q.dy)));
  q.objA = (den.x > 0.f) & (ro.x <= rs.x);  // false for NaN (edge-on disks)
  q.objB = (den.y > 0.f) & (ro.y <= rs.y);
  q.rho = sel2(q.objA, q.objB, ro, rs);
  const float2 x = mul2(bc(kNegHalfLog2e), q.rho);
  const float2 a = mul2(bc(opac), make_float2(ex2_approx(x.x), ex2_approx(x.y)));
  q.alpha = make_float2(fminf(set.alpha_max, a.x), fminf(set.alpha_max, a.y));
  q.hitA = (q.rho.x <= set.rho_max) & (q.alpha.x >= set.alpha_min);
  q.hitB = (q.rho.y <= set.rho_max) & (q.alpha.y >= set.alpha_min);
  return q;
}

// ---------------------------------------------------------------------------
// Forward.

// Shared-memory staging area of one CTA.
struct FwdSmem {
  float4 s0[kBatch], s1[kBatch], s2[kBatch], s3[kBatch], s4[kBatch], s5[kBatch];
  uint16_t sm[kBatch];
  uint8_t list[kThreads / 32][4][kListStride<kBatch>];
  unsigned long long tot[2];
};

// Running sums of one pixel.  Z is accumulated relative to zr, the depth of
// the first blended pair: sum w (z - zr) keeps the distortion terms z A - Z
// free of the cancellation between depths of hundreds of metres (both are
// invariant under a common shift of z), and sum w z = sum w (z - zr) + zr A.
struct FwdPix {
  float T, C0, C1, C2, A, Zs, zr, I, N0, N1, N2, D, M;
  int cnt, lastpos, medpos;
};

__device__ __forceinline__ void fwd_init(FwdPix& p) {
  p.T = 1.f;
  p.C0 = p.C1 = p.C2 = p.A = p.Zs = p.zr = p.I = p.N0 = p.N1 = p.N2 = p.D = p.M = 0.f;
  p.cnt = 0;
  p.lastpos = 0;
  p.medpos = -1;
}

// The same for a thread's two pixels.  evaluated counts the entries visited
// before a pixel was done.
struct FwdPair {
  float2 T, C0, C1, C2, A, Zs, zr, I, N0, N1, N2, D, M;
  int cntA, cntB, lastA, lastB, medA, medB;
  unsigned evaluated;
  bool doneA, doneB;
  __device__ __forceinline__ FwdPix a() const {
    return {T.x, C0.x, C1.x, C2.x, A.x, Zs.x, zr.x, I.x, N0.x, N1.x, N2.x, D.x, M.x, cntA, lastA, medA};
  }
  __device__ __forceinline__ FwdPix b() const {
    return {T.y, C0.y, C1.y, C2.y, A.y, Zs.y, zr.y, I.y, N0.y, N1.y, N2.y, D.y, M.y, cntB, lastB, medB};
  }
};

__device__ __forceinline__ void fwd_init(FwdPair& p, bool insideA, bool insideB) {
  p.T = bc(1.f);
  p.C0 = p.C1 = p.C2 = p.A = p.Zs = p.zr = p.I = p.N0 = p.N1 = p.N2 = p.D = p.M = bc(0.f);
  p.cntA = p.cntB = p.lastA = p.lastB = 0;
  p.medA = p.medB = -1;
  p.evaluated = 0;
  p.doneA = !insideA;
  p.doneB = !insideB;
}

// One list entry (position pos, already evaluated as q) against the two
// pixels.  Branch-free: a pair that is not blended updates the sums with alpha
// 0 (and a finite depth), which leaves them unchanged.  kPos: also the
// positions of the last blended and the median entry.  kFixedRef: zr is given.
// Returns whether a pixel stopped at this entry.
template <bool kFixedRef, bool kPos>
__device__ __forceinline__ bool fwd_step(FwdPair& p, const Pair& q, float4 e2, float4 e3, int pos, const SetDev& set,
                                         bool* stopA, bool* stopB) {
  const float2 one = bc(1.f);
  const float2 Tn = mul2(p.T, fma2(neg2(q.alpha), one, one));
  const bool hA = !p.doneA & q.hitA, hB = !p.doneB & q.hitB;
  *stopA = hA & (Tn.x < set.T_min);
  *stopB = hB & (Tn.y < set.T_min);
  const bool blA = hA & !(Tn.x < set.T_min), blB = hB & !(Tn.y < set.T_min);
  const float2 al = sel2(blA, blB, q.alpha, bc(0.f));
  const float2 w = mul2(al, p.T);
  const float2 z = sel2(q.objA, q.objB, mul2(bc(e2.x), q.rden), bc(e2.x));
  p.C0 = fma2(w, bc(e2.z), p.C0);
  p.C1 = fma2(w, bc(e2.w), p.C1);
  p.C2 = fma2(w, bc(e3.x), p.C2);
  if constexpr (!kFixedRef) p.zr = sel2(blA & (p.cntA == 0), blB & (p.cntB == 0), z, p.zr);
  const float2 zs = add2(z, neg2(p.zr));
  p.D = fma2(add2(w, w), fma2(zs, p.A, neg2(p.Zs)), p.D);
  p.A = add2(p.A, w);
  p.Zs = fma2(w, zs, p.Zs);
  p.I = fma2(w, rcp2(z), p.I);
  p.N0 = fma2(w, bc(e3.y), p.N0);
  p.N1 = fma2(w, bc(e3.z), p.N1);
  p.N2 = fma2(w, bc(e3.w), p.N2);
  const bool mA = blA & (p.T.x > 0.5f), mB = blB & (p.T.y > 0.5f);
  p.M = sel2(mA, mB, z, p.M);
  if constexpr (kPos) {
    p.medA = mA ? pos : p.medA;
    p.medB = mB ? pos : p.medB;
    p.lastA = blA ? pos + 1 : p.lastA;
    p.lastB = blB ? pos + 1 : p.lastB;
  }
  p.T = mul2(p.T, fma2(neg2(al), one, one));
  p.cntA += blA ? 1 : 0;
  p.cntB += blB ? 1 : 0;
  return *stopA | *stopB;
}

// A lane group's walk over its list of one batch (list positions b0 + k),
// front to back, until both of the thread's pixels are done.
template <bool kFixedRef, bool kPos>
__device__ __forceinline__ void fwd_walk(FwdPair& p, const FwdSmem& sh, const uint8_t* list, int glen, int b0, float lx,
                                         float2 ly, const SetDev& set) {
  if (p.doneA && p.doneB) return;
  int k = list[0];
  for (int i = 0; i < glen; ++i) {
    const float4 e0 = sh.s0[k], e1 = sh.s1[k], e2 = sh.s2[k], e3 = sh.s3[k], e4 = sh.s4[k], e5 = sh.s5[k];
    const int pos = b0 + k;
    k = list[i + 1];  // past the end: a byte of padding, not used
    const Pair q = eval_pair(lx, ly, e0, e1, e4, e5, e2.y, set);
    bool stopA, stopB;
    if (fwd_step<kFixedRef, kPos>(p, q, e2, e3, pos, set, &stopA, &stopB)) {  // once per pixel
      p.evaluated += (stopA ? i + 1 : 0) + (stopB ? i + 1 : 0);
      p.doneA = p.doneA || stopA;
      p.doneB = p.doneB || stopB;
      if (p.doneA && p.doneB) return;
    }
  }
  p.evaluated += (p.doneA ? 0 : glen) + (p.doneB ? 0 : glen);
}

__device__ __forceinline__ void fwd_store(const FwdPix& p, const CamDev& cam, const SetDev& set, int px,
                                          int py, float* __restrict__ out, int32_t* __restrict__ n_contrib,
                                          int32_t* __restrict__ last, int32_t* __restrict__ med) {
  if (px >= cam.W || py >= cam.H) return;
  const size_t HW = (size_t)cam.W * cam.H;
  const size_t i = (size_t)py * cam.W + px;
  out[i] = p.C0 + p.T * set.bg[0];
  out[HW + i] = p.C1 + p.T * set.bg[1];
  out[2 * HW + i] = p.C2 + p.T * set.bg[2];
  out[3 * HW + i] = p.A;
  out[4 * HW + i] = fmaf(p.zr, p.A, p.Zs);
  out[5 * HW + i] = p.I;
  out[6 * HW + i] = p.M;
  out[7 * HW + i] = p.N0;
  out[8 * HW + i] = p.N1;
  out[9 * HW + i] = p.N2;
  out[10 * HW + i] = p.D;
  out[11 * HW + i] = p.T;
  if (n_contrib) n_contrib[i] = p.cnt;
  if (last) last[i] = p.lastpos;
  if (med) med[i] = p.medpos;
}

// Stage nb entries of a tile's list from position base on (the entries that
// reach no pixel block of the tile leave their slot as it is: no list has it).
__device__ __forceinline__ void stage_batch(FwdSmem& sh, const float4* __restrict__ rec,
                                            const uint16_t* __restrict__ masks, const uint32_t* __restrict__ vals,
                                            int base, int nb, int tx0, int ty0) {
  for (int t = threadIdx.x; t < nb; t += kThreads) {
    const uint16_t m = masks[base + t];
    sh.sm[t] = m;
    if (m == 0u) continue;
    const Staged e = stage_entry(rec, vals[base + t], tx0, ty0);
    sh.s0[t] = e.s0;
    sh.s1[t] = e.s1;
    sh.s2[t] = e.s2;
    sh.s3[t] = e.s3;
    sh.s4[t] = e.s4;
    sh.s5[t] = e.s5;
  }
}

// Forward blend of tile (bx, by) of one view by the whole CTA.
template <bool kPos>
__device__ __forceinline__ void blend_fwd_tile(
    FwdSmem& sh, const CamDev& cam, const SetDev& set, const float4* __restrict__ rec,
    const uint16_t* __restrict__ masks, const uint32_t* __restrict__ vals, const int2* __restrict__ ranges,
    float* __restrict__ out, int32_t* __restrict__ n_contrib, int32_t* __restrict__ last,
    int32_t* __restrict__ med, unsigned long long* __restrict__ counters, int bx, int by, int lseg = 0) {
  const int tile = by * cam.tiles_x + bx;
  const int tx0 = bx * kTile, ty0 = by * kTile;
  const int lxi = local_x(threadIdx.x), lyi = local_y(threadIdx.x);
  const int px = tx0 + lxi, pyA = ty0 + lyi, pyB = pyA + kRowStep;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const float lx = (float)lxi + 0.5f;
  const float2 ly = make_float2((float)lyi + 0.5f, (float)(lyi + kRowStep) + 0.5f);
  const int2 rg = ranges[tile];
  const int len = rg.y - rg.x;
  if (lseg > 0 && len > lseg) return;  // a long list: composited in segments
  FwdPair p;
  fwd_init(p, px < cam.W && pyA < cam.H, px < cam.W && pyB < cam.H);
  for (int b0 = 0; b0 < len; b0 += kBatch) {
    if (__syncthreads_count(p.doneA && p.doneB) == kThreads) break;
    const int nb = min(kBatch, len - b0);
    stage_batch(sh, rec, masks, vals, rg.x + b0, nb, tx0, ty0);
    __syncthreads();
    const int glen = group_lists<kBatch>(sh.sm, nb, warp, lane, sh.list[warp]);
    fwd_walk<false, kPos>(p, sh, sh.list[warp][lane >> 3], glen, b0, lx, ly, set);
  }
  fwd_store(p.a(), cam, set, px, pyA, out, n_contrib, last, med);
  fwd_store(p.b(), cam, set, px, pyB, out, n_contrib, last, med);
  if (counters) {
    // per-tile totals of evaluated and blended pairs (performance counters)
    unsigned long long* tot = sh.tot;
    if (threadIdx.x == 0) tot[0] = tot[1] = 0ull;
    __syncthreads();
    unsigned e = p.evaluated, c = (unsigned)(p.cntA + p.cntB);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      e += __shfl_xor_sync(0xffffffffu, e, o);
      c += __shfl_xor_sync(0xffffffffu, c, o);
    }
    if (lane == 0) {
      atomicAdd(&tot[0], (unsigned long long)e);
      atomicAdd(&tot[1], (unsigned long long)c);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      atomicAdd(&counters[0], tot[0]);
      atomicAdd(&counters[1], tot[1]);
    }
  }
}

// One CTA per tile; block b takes tile order[b] (longest lists first).
template <bool kPos>
__global__ void __launch_bounds__(kThreads, 5) blend_fwd_kernel(
    CamDev cam, SetDev set, const uint32_t* __restrict__ order, const float4* __restrict__ rec,
    const uint16_t* __restrict__ masks, const uint32_t* __restrict__ vals, const int2* __restrict__ ranges,
    float* __restrict__ out, int32_t* __restrict__ n_contrib, int32_t* __restrict__ last,
    int32_t* __restrict__ med, unsigned long long* __restrict__ counters, int lseg) {
  __shared__ FwdSmem sh;
  const int t = order ? (int)order[blockIdx.x] : (int)blockIdx.x;
  blend_fwd_tile<kPos>(sh, cam, set, rec, masks, vals, ranges, out, n_contrib, last, med, counters,
                 t % cam.tiles_x, t / cam.tiles_x, lseg);
}

// ---------------------------------------------------------------------------
// Long lists, composited in segments.
//
// When an image has too few tiles to fill the GPU and some tiles carry long
// lists (a small view of a large scene), a tile's list is cut into segments
// of lseg entries that separate CTAs process:
//   1. seg_trans_kernel: per segment and pixel, the product of (1 - alpha)
//      over the segment's pairs that pass the support and cutoff tests (no
//      stop).  Below T_min the product's value decides nothing any more, so a
//      segment ends once it is there for all pixels.  The same launch
//      composites the tiles with short lists whole: one after the other, the
//      two left the GPU half empty;
//   2. seg_blend_kernel: per segment, the pixel enters with the product of
//      the segments in front (the transmittance it would have there had
//      nothing stopped) and composites the segment with the forward's rules,
//      the stop included.  A pixel that stopped in an earlier segment enters
//      below T_min and is done;
//   3. seg_merge_kernel: per tile and pixel, the segments are combined in
//      order.  Sums add; the distortion adds the cross terms
//      2 (A_front Zs_seg - Zs_front A_seg) (depths relative to one reference,
//      the tile's first centre depth); the median comes from the last
//      segment that has one; T and the stop from the segment where blending
//      ended.
// The result equals the one-CTA compositing up to the rounding of T's
// products (decisions within a hair of a threshold may differ).

struct SegPart {
  float4 f0;  // C0, C1, C2, A
  float4 f1;  // Zs (relative to the reference), I, N0, N1
  float4 f2;  // N2, D, M, T after the segment
  int4 f3;    // median position, count, last position, stopped
};

// Segment b of the split tiles: its tile and its index within the tile.
__device__ __forceinline__ bool seg_of(const uint32_t* seg_tile, const uint32_t* seg_idx, const uint32_t* nseg,
                                       int b, int* tile, int* s) {
  if ((uint32_t)b >= *nseg) return false;
  *tile = (int)seg_tile[b];
  *s = (int)seg_idx[b];
  return true;
}

__global__ void __launch_bounds__(kThreads, 5) seg_trans_kernel(
    CamDev cam, SetDev set, const uint32_t* __restrict__ order, const float4* __restrict__ rec,
    const uint16_t* __restrict__ masks, const uint32_t* __restrict__ vals, const int2* __restrict__ ranges,
    float* __restrict__ out, int32_t* __restrict__ n_contrib, int32_t* __restrict__ last, int32_t* __restrict__ med,
    unsigned long long* __restrict__ counters, int lseg, const uint32_t* __restrict__ seg_tile,
    const uint32_t* __restrict__ seg_idx, const uint32_t* __restrict__ nseg, float* __restrict__ trans) {
  __shared__ FwdSmem sh;
  const int ntiles = cam.tiles_x * cam.tiles_y;
  if ((int)blockIdx.x < ntiles) {
    const int t = order ? (int)order[blockIdx.x] : (int)blockIdx.x;
    blend_fwd_tile<true>(sh, cam, set, rec, masks, vals, ranges, out, n_contrib, last, med, counters, t % cam.tiles_x,
                         t / cam.tiles_x, lseg);
    return;
  }
  const int seg = (int)blockIdx.x - ntiles;
  int tile, s;
  if (!seg_of(seg_tile, seg_idx, nseg, seg, &tile, &s)) return;
  const int tx0 = (tile % cam.tiles_x) * kTile, ty0 = (tile / cam.tiles_x) * kTile;
  const int lxi = local_x(threadIdx.x), lyi = local_y(threadIdx.x);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const float lx = (float)lxi + 0.5f;
  const float2 ly = make_float2((float)lyi + 0.5f, (float)(lyi + kRowStep) + 0.5f);
  const int2 rg = ranges[tile];
  const int e0 = s * lseg, e1 = min(rg.y - rg.x, e0 + lseg);
  // pixels outside the image enter no product
  const bool inA = tx0 + lxi < cam.W && ty0 + lyi < cam.H, inB = tx0 + lxi < cam.W && ty0 + lyi + kRowStep < cam.H;
  float2 T = make_float2(inA ? 1.f : 0.f, inB ? 1.f : 0.f);
  for (int b0 = e0; b0 < e1; b0 += kBatch) {
    const int nb = min(kBatch, e1 - b0);
    const bool below = !(T.x >= set.T_min) && !(T.y >= set.T_min);
    if (__syncthreads_count(below) == kThreads) break;
    stage_batch(sh, rec, masks, vals, rg.x + b0, nb, tx0, ty0);
    __syncthreads();
    if (__all_sync(0xffffffffu, below)) continue;
    int glen = group_lists<kBatch>(sh.sm, nb, warp, lane, sh.list[warp]);
    if (below) glen = 0;
    const uint8_t* list = sh.list[warp][lane >> 3];
    for (int i = 0; i < glen; ++i) {
      const int k = list[i];
      const Pair q = eval_pair(lx, ly, sh.s0[k], sh.s1[k], sh.s4[k], sh.s5[k], sh.s2[k].y, set);
      const float2 al = sel2(q.hitA, q.hitB, q.alpha, bc(0.f));
      T = mul2(T, fma2(neg2(al), bc(1.f), bc(1.f)));
    }
  }
  trans[(size_t)seg * kTilePix + threadIdx.x] = T.x;
  trans[(size_t)seg * kTilePix + kThreads + threadIdx.x] = T.y;
}

__device__ __forceinline__ void seg_store(const FwdPix& p, bool stopped, SegPart* __restrict__ part, int slot) {
  SegPart q;
  q.f0 = make_float4(p.C0, p.C1, p.C2, p.A);
  q.f1 = make_float4(p.Zs, p.I, p.N0, p.N1);
  q.f2 = make_float4(p.N2, p.D, p.M, p.T);
  q.f3 = make_int4(p.medpos, p.cnt, p.lastpos, stopped ? 1 : 0);
  part[slot] = q;
}

__global__ void __launch_bounds__(kThreads, 5) seg_blend_kernel(
    CamDev cam, SetDev set, const float4* __restrict__ rec, const uint16_t* __restrict__ masks,
    const uint32_t* __restrict__ vals, const int2* __restrict__ ranges, int lseg,
    const uint32_t* __restrict__ seg_tile, const uint32_t* __restrict__ seg_idx, const uint32_t* __restrict__ nseg,
    const float* __restrict__ trans, SegPart* __restrict__ part, unsigned long long* __restrict__ counters) {
  __shared__ FwdSmem sh;
  int tile, s;
  if (!seg_of(seg_tile, seg_idx, nseg, blockIdx.x, &tile, &s)) return;
  const int tx0 = (tile % cam.tiles_x) * kTile, ty0 = (tile / cam.tiles_x) * kTile;
  const int lxi = local_x(threadIdx.x), lyi = local_y(threadIdx.x);
  const int px = tx0 + lxi, pyA = ty0 + lyi, pyB = pyA + kRowStep;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const float lx = (float)lxi + 0.5f;
  const float2 ly = make_float2((float)lyi + 0.5f, (float)(lyi + kRowStep) + 0.5f);
  const int2 rg = ranges[tile];
  const int e0 = s * lseg, e1 = min(rg.y - rg.x, e0 + lseg);
  const bool inA = px < cam.W && pyA < cam.H, inB = px < cam.W && pyB < cam.H;
  FwdPair p;
  fwd_init(p, inA, inB);
  // transmittance in front: the segments before this one (contiguous)
  const int first = (int)blockIdx.x - s;
  for (int q = 0; q < s; ++q) {
    p.T.x *= trans[(size_t)(first + q) * kTilePix + threadIdx.x];
    p.T.y *= trans[(size_t)(first + q) * kTilePix + kThreads + threadIdx.x];
  }
  p.doneA = p.doneA || p.T.x < set.T_min;
  p.doneB = p.doneB || p.T.y < set.T_min;
  p.zr = bc(rec[(size_t)vals[rg.x] * kRecF4 + 2].z);  // the tile's first centre depth
  for (int b0 = e0; b0 < e1; b0 += kBatch) {
    if (__syncthreads_count(p.doneA && p.doneB) == kThreads) break;
    const int nb = min(kBatch, e1 - b0);
    stage_batch(sh, rec, masks, vals, rg.x + b0, nb, tx0, ty0);
    __syncthreads();
    const int glen = group_lists<kBatch>(sh.sm, nb, warp, lane, sh.list[warp]);
    fwd_walk<true, true>(p, sh, sh.list[warp][lane >> 3], glen, b0, lx, ly, set);
  }
  SegPart* pp = part + (size_t)blockIdx.x * kTilePix;
  seg_store(p.a(), inA && p.doneA, pp, threadIdx.x);
  seg_store(p.b(), inB && p.doneB, pp, kThreads + threadIdx.x);
  if (counters) {
    unsigned e = p.evaluated, c = (unsigned)(p.cntA + p.cntB);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      e += __shfl_xor_sync(0xffffffffu, e, o);
      c += __shfl_xor_sync(0xffffffffu, c, o);
    }
    if ((threadIdx.x & 31) == 0) {
      atomicAdd(&counters[0], (unsigned long long)e);
      atomicAdd(&counters[1], (unsigned long long)c);
    }
  }
}

// Combine the segments of one pixel in order (slot = its index within the
// segment records).
__device__ __forceinline__ FwdPix seg_merge_pixel(const SegPart* __restrict__ part, int first, int nseg_tile,
                                                  int slot, float zref) {
  FwdPix p;
  fwd_init(p);
  p.zr = zref;
  bool stopped = false;
  for (int q = 0; q < nseg_tile && !stopped; ++q) {
    const SegPart g = part[(size_t)(first + q) * kTilePix + slot];
    p.C0 += g.f0.x;
    p.C1 += g.f0.y;
    p.C2 += g.f0.z;
    p.D += g.f2.y + 2.f * (p.A * g.f1.x - p.Zs * g.f0.w);
    p.A += g.f0.w;
    p.Zs += g.f1.x;
    p.I += g.f1.y;
    p.N0 += g.f1.z;
    p.N1 += g.f1.w;
    p.N2 += g.f2.x;
    if (g.f3.x >= 0) {
      p.M = g.f2.z;
      p.medpos = g.f3.x;
    }
    if (g.f3.y > 0) p.lastpos = g.f3.z;
    p.cnt += g.f3.y;
    p.T = g.f2.w;
    stopped = g.f3.w != 0;
  }
  return p;
}

__global__ void __launch_bounds__(kThreads) seg_merge_kernel(
    CamDev cam, SetDev set, const float4* __restrict__ rec, const uint32_t* __restrict__ vals,
    const int2* __restrict__ ranges, const uint32_t* __restrict__ segcnt, const uint32_t* __restrict__ seg_tile,
    const uint32_t* __restrict__ seg_idx, const uint32_t* __restrict__ nseg, const SegPart* __restrict__ part,
    float* __restrict__ out, int32_t* __restrict__ n_contrib, int32_t* __restrict__ last,
    int32_t* __restrict__ med) {
  int tile, s;
  if (!seg_of(seg_tile, seg_idx, nseg, blockIdx.x, &tile, &s) || s != 0) return;
  const int tx0 = (tile % cam.tiles_x) * kTile, ty0 = (tile / cam.tiles_x) * kTile;
  const int lxi = local_x(threadIdx.x), lyi = local_y(threadIdx.x);
  const int px = tx0 + lxi, pyA = ty0 + lyi, pyB = pyA + kRowStep;
  const int2 rg = ranges[tile];
  const float zref = rec[(size_t)vals[rg.x] * kRecF4 + 2].z;
  const int ns = (int)segcnt[tile];
  const FwdPix a = seg_merge_pixel(part, blockIdx.x, ns, threadIdx.x, zref);
  const FwdPix b = seg_merge_pixel(part, blockIdx.x, ns, kThreads + threadIdx.x, zref);
  fwd_store(a, cam, set, px, pyA, out, n_contrib, last, med);
  fwd_store(b, cam, set, px, pyB, out, n_contrib, last, med);
}

// Segments per tile (0 for tiles composited whole).
__global__ void seg_count_kernel(const int2* __restrict__ ranges, int ntiles, int lseg, uint32_t* __restrict__ segcnt) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= ntiles) return;
  const int len = ranges[t].y - ranges[t].x;
  segcnt[t] = len > lseg ? (uint32_t)((len + lseg - 1) / lseg) : 0u;
}

__global__ void seg_list_kernel(const uint32_t* __restrict__ segcnt, const uint32_t* __restrict__ segoff, int ntiles,
                                uint32_t* __restrict__ seg_tile, uint32_t* __restrict__ seg_idx) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= ntiles) return;
  const uint32_t c = segcnt[t], o = segoff[t];
  for (uint32_t q = 0; q < c; ++q) {
    seg_tile[o + q] = (uint32_t)t;
    seg_idx[o + q] = q;
  }
}

// Persistent forward blend over the tiles of several views (serving): each
// CTA takes (view, tile) work items from a device counter until all tiles
// of all views in the batch are done; views of different sizes and scenes
// share one launch.
__global__ void __launch_bounds__(kThreads, 5) blend_fwd_batched_kernel(BlendBatch batch) {
  __shared__ FwdSmem sh;
  __shared__ int item;
  for (;;) {
    __syncthreads();
    if (threadIdx.x == 0) item = (int)atomicAdd(batch.counter, 1u);
    __syncthreads();
    const int t = item;
    if (t >= batch.total_tiles) break;
    int j = 0;
    while (j + 1 < batch.njobs && batch.job[j + 1].tile_begin <= t) ++j;
    const BlendJob& jb = batch.job[j];
    const int local = t - jb.tile_begin;
    blend_fwd_tile<false>(sh, jb.cam, jb.set, jb.rec, jb.masks, jb.vals, jb.ranges, jb.out, jb.n_contrib,
                   nullptr, nullptr, batch.work, local % jb.cam.tiles_x, local / jb.cam.tiles_x);
  }
}

// ---------------------------------------------------------------------------
// Backward.

constexpr int kMaxSets = 3;
// Per-entry gradient vector, the surfel's gradient row (kRow* in
// gs2d_internal.cuh): d Ji, d e, the screen-space gradient of set 0, the depth
// term of the centre gradient, d p_z, opacity times d opacity, d rgb, the
// screen-space gradients of sets 1 and 2, and in the general layout d normal.
// The loss layout (set 0 on colour and inverse depth only, later sets on
// colour) has no d normal.  d c is not summed from its own terms: per pair it
// is set 0's screen gradient plus, on the object-space branch, the term of the
// depth z = p_z / (1 + e.d) through d, (d rden / d d) p_z dz = -e p_z rden^2 dz;
// so d c = (screen gradient of set 0) + e * (sum of p_z rden^2 dz), formed once
// per surfel by the preprocess's backward, and d alpha / d opacity = alpha /
// opacity, divided there.
//
// The reduce-scatter leaves lane r of a group the sums of up to three
// consecutive values; nat() places the vector so that the groups' first,
// second and third values are consecutive in the row.
template <bool kLoss>
struct Layout {
  static constexpr int kN = kLoss ? kRowLoss : kRowAll;
  // first value of lane r (the halving of kN: 3 2 3 1 3 2 3 1, 3 3 3 2 3 3 3 1)
  __host__ __device__ static constexpr int start(int r) {
    return kLoss ? 9 * (r >> 2) + 5 * ((r >> 1) & 1) + 3 * (r & 1) : 11 * (r >> 2) + 6 * ((r >> 1) & 1) + 3 * (r & 1);
  }
  // the row's value at lane r's i-th place, -1 when it has none
  __host__ __device__ static constexpr int at(int r, int i) {
    if (i == 0) return r;
    if (kLoss) {
      if (i == 1) return (r & 3) == 3 ? -1 : 8 + r - (r > 3 ? 1 : 0);
      return (r & 1) ? -1 : 14 + (r >> 1);
    }
    if (i == 1) return r == 7 ? -1 : 8 + r;
    return (r & 3) == 3 ? -1 : 15 + r - (r > 3 ? 1 : 0);
  }
  __host__ __device__ static constexpr int nat(int m) {
    for (int r = 0; r < 8; ++r)
      for (int i = 0; i < 3; ++i)
        if (at(r, i) == m) return start(r) + i;
    return -1;
  }
};
constexpr bool layout_is_permutation(bool loss) {
  const int n = loss ? kRowLoss : kRowAll;
  uint32_t seen = 0;
  for (int m = 0; m < n; ++m) {
    const int v = loss ? Layout<true>::nat(m) : Layout<false>::nat(m);
    if (v < 0 || v >= n || ((seen >> v) & 1u)) return false;
    seen |= 1u << v;
  }
  return true;
}
static_assert(layout_is_permutation(true) && layout_is_permutation(false), "one place per value");

// Balanced reduce-scatter of N values over a lane group of eight: at each
// halving level the lanes whose bit is clear keep the first ceil(N/2) values
// and the others the rest, exchanging the halves they do not keep (17
// shuffles for 18 values, and the warp's four groups reduce four entries at
// once).  Afterwards v[0..2] hold the group's sums of values start(r) + 0..2.
constexpr int kGroup = 8;
template <int O, int N>
__device__ __forceinline__ void rs_level(float* v, int lane) {
  constexpr int L = (N + 1) / 2, H = N - L;
  const bool up = (lane & O) != 0;
#pragma unroll
  for (int i = 0; i < L; ++i) {
    const float hi = (i < H) ? v[L + i] : 0.f;
    const float send = up ? v[i] : hi;
    const float keep = up ? hi : v[i];
    v[i] = keep + __shfl_xor_sync(0xffffffffu, send, O);
  }
  if constexpr (O > 1) rs_level<O / 2, L>(v, lane);
}

// State of the reverse replay of a thread's two pixels (the halves of each
// pair): transmittance, suffix sums S of each adjoint set, the pixels'
// adjoints, and (general layout) the running opacity A and depth sum Z with
// their final values for the distortion; gD2 is twice the distortion's adjoint.
struct BwdPix {
  float2 T, A, Z, Af, Zf;
  float2 S[kMaxSets];
  float2 gC[kMaxSets][3];
  float2 gA, gZ, gI, gMed, gD2, gN0, gN1, gN2;
  int lastA, lastB, medA, medB;
};

// One half of the state: the pixel at index pix (nothing when outside).
struct BwdInit {
  float T, A, Z, S[kMaxSets], gC[kMaxSets][3], gA, gZ, gI, gMed, gD2, gN0, gN1, gN2;
  int last, med;
};

template <bool kLoss>
__device__ __forceinline__ BwdInit bwd_load(bool inside, size_t pix, size_t HW, const float* __restrict__ out,
                                            const int32_t* __restrict__ last, const int32_t* __restrict__ med,
                                            const AdjDev& adj, const SetDev& set) {
  BwdInit p;
  p.T = 1.f;
  p.A = p.Z = 0.f;
  p.gA = p.gZ = p.gI = p.gMed = p.gD2 = p.gN0 = p.gN1 = p.gN2 = 0.f;
  p.last = 0;
  p.med = -1;
#pragma unroll
  for (int s = 0; s < kMaxSets; ++s) {
    p.gC[s][0] = p.gC[s][1] = p.gC[s][2] = 0.f;
    p.S[s] = 0.f;
  }
  if (!inside) return p;
  p.last = last[pix];
  p.T = out[11 * HW + pix];
#pragma unroll
  for (int s = 0; s < kMaxSets; ++s) {
    if (s >= adj.n_sets) break;
    const float* a = adj.set[s];
    const uint32_t m = adj.mask[s];
#pragma unroll
    for (int c = 0; c < 3; ++c) p.gC[s][c] = (m >> c) & 1u ? a[c * HW + pix] : 0.f;
    p.S[s] = p.T * (p.gC[s][0] * set.bg[0] + p.gC[s][1] * set.bg[1] + p.gC[s][2] * set.bg[2]);
  }
  const float* a = adj.set[0];
  const uint32_t m = adj.mask[0];
  if (m & (1u << 5)) p.gI = a[5 * HW + pix];
  if constexpr (!kLoss) {
    p.med = med[pix];
    p.A = out[3 * HW + pix];
    p.Z = out[4 * HW + pix];
    if (m & (1u << 3)) p.gA = a[3 * HW + pix];
    if (m & (1u << 4)) p.gZ = a[4 * HW + pix];
    if (m & (1u << 6)) p.gMed = a[6 * HW + pix];
    if (m & (1u << 7)) p.gN0 = a[7 * HW + pix];
    if (m & (1u << 8)) p.gN1 = a[8 * HW + pix];
    if (m & (1u << 9)) p.gN2 = a[9 * HW + pix];
    if (m & (1u << 10)) p.gD2 = 2.f * a[10 * HW + pix];
  }
  return p;
}

__device__ __forceinline__ void bwd_init(BwdPix& p, const BwdInit& a, const BwdInit& b) {
  p.T = make_float2(a.T, b.T);
  p.A = p.Af = make_float2(a.A, b.A);
  p.Z = p.Zf = make_float2(a.Z, b.Z);
#pragma unroll
  for (int s = 0; s < kMaxSets; ++s) {
    p.S[s] = make_float2(a.S[s], b.S[s]);
#pragma unroll
    for (int c = 0; c < 3; ++c) p.gC[s][c] = make_float2(a.gC[s][c], b.gC[s][c]);
  }
  p.gA = make_float2(a.gA, b.gA);
  p.gZ = make_float2(a.gZ, b.gZ);
  p.gI = make_float2(a.gI, b.gI);
  p.gMed = make_float2(a.gMed, b.gMed);
  p.gD2 = make_float2(a.gD2, b.gD2);
  p.gN0 = make_float2(a.gN0, b.gN0);
  p.gN1 = make_float2(a.gN1, b.gN1);
  p.gN2 = make_float2(a.gN2, b.gN2);
  p.lastA = a.last;
  p.lastB = b.last;
  p.medA = a.med;
  p.medB = b.med;
}

__device__ __forceinline__ float hsum(float2 x) { return x.x + x.y; }
__device__ __forceinline__ float dot2(float2 a, float2 b) { return fmaf(a.y, b.y, a.x * b.x); }

// Gradients of the thread's two pairs at list position k, added up into v
// (gradient-vector layout), and the pixels' replay state moved past the entry.
// Branch-free.  A pair that was not blended (or lies past the pixel's last
// blended entry) has hit false: with alpha 0 on the screen-space branch every
// term is a finite zero and the pixel's state passes through.  The screen
// branch is the object branch with (nu, nv) = 0 and rden = 1 (then u = v = 0,
// z = p_z and only the depth's chain through e.d has to be masked) plus the
// term sinv d of rho_scr.
template <bool kLoss>
__device__ __forceinline__ void bwd_pair(BwdPix& p, const Pair& q, bool hitA, bool hitB, float4 e0, float4 e1,
                                         float4 e2, float4 e3, int k, int nsets, const SetDev& set, float* v) {
  using LY = Layout<kLoss>;
  const float2 one = bc(1.f), zero = bc(0.f);
  const float2 al = sel2(hitA, hitB, q.alpha, zero);
  const bool oA = hitA & q.objA, oB = hitB & q.objB;
  const float2 rd = sel2(oA, oB, q.rden, one);
  const float2 nu = sel2(oA, oB, q.nu, zero), nv = sel2(oA, oB, q.nv, zero);
  const float2 rom = rcp2(fma2(neg2(al), one, one));
  p.T = sel2(hitA, hitB, mul2(p.T, rom), p.T);  // transmittance before this pair
  const float2 w = mul2(al, p.T);
  const float2 z = mul2(bc(e2.x), rd);
  const float2 rz = rcp2(z);
  float2 dLdw = fma2(p.gC[0][0], bc(e2.z), mul2(p.gC[0][1], bc(e2.w)));
  dLdw = fma2(p.gI, rz, fma2(p.gC[0][2], bc(e3.x), dLdw));
  float2 dzv = mul2(mul2(mul2(neg2(w), p.gI), rz), rz);
  if constexpr (!kLoss) {
    const float2 Ap = add2(p.A, neg2(w)), Zp = fma2(neg2(w), z, p.Z);  // in front of this pair
    const float2 Ab = add2(p.Af, neg2(p.A)), Zb = add2(p.Zf, neg2(p.Z));  // behind it
    const float2 dD = fma2(neg2(z), Ab, add2(fma2(z, Ap, neg2(Zp)), Zb));
    dLdw = fma2(p.gZ, z, add2(dLdw, p.gA));
    dLdw = fma2(p.gN2, bc(e3.w), fma2(p.gN1, bc(e3.z), fma2(p.gN0, bc(e3.y), dLdw)));
    dLdw = fma2(p.gD2, dD, dLdw);
    dzv = fma2(w, fma2(p.gD2, add2(Ap, neg2(Ab)), p.gZ), dzv);
    dzv = add2(dzv, sel2(hitA & (k == p.medA), hitB & (k == p.medB), p.gMed, zero));
    p.A = Ap;
    p.Z = Zp;
  }
  // alpha -> rho (zero where alpha is clamped at alpha_max): d alpha / d rho =
  // -alpha / 2; every derivative of rho below carries a factor 2, so
  // nd = -2 dL / d rho = dL/dalpha alpha
  const float2 am = make_float2(al.x < set.alpha_max ? al.x : 0.f, al.y < set.alpha_max ? al.y : 0.f);
  float2 nd[kMaxSets];
  nd[0] = mul2(fma2(p.T, dLdw, neg2(mul2(p.S[0], rom))), am);
  p.S[0] = fma2(w, dLdw, p.S[0]);
#pragma unroll
  for (int s = 1; s < kMaxSets; ++s) {
    if (s < nsets) {
      const float2 dw = fma2(p.gC[s][2], bc(e3.x), fma2(p.gC[s][0], bc(e2.z), mul2(p.gC[s][1], bc(e2.w))));
      nd[s] = mul2(fma2(p.T, dw, neg2(mul2(p.S[s], rom))), am);
      p.S[s] = fma2(w, dw, p.S[s]);
    } else {
      nd[s] = zero;
    }
  }
  // rho = u^2 + v^2 with (u, v) = (nu, nv) rden, z = p_z rden;
  // rx, ry are half of d rho / d d
  const float2 u = mul2(nu, rd), vv = mul2(nv, rd);
  const float2 up = mul2(u, rd), vp = mul2(vv, rd);
  const float2 c1 = fma2(u, up, mul2(vv, vp));
  const float2 r2d = mul2(rd, rd), dzp = sel2(oA, oB, mul2(dzv, bc(e2.x)), zero);
  const float2 zr2 = mul2(dzp, r2d);
  const float2 dnu = mul2(up, neg2(nd[0])), dnv = mul2(vp, neg2(nd[0]));
  // d L / d rden, then through rden = 1 / (1 + e.d)
  const float2 dden = fma2(nd[0], c1, neg2(zr2));
  const float2 ks = sel2(oA, oB, zero, bc(set.sinv));
  const float2 rx = fma2(ks, bc(q.dx), fma2(c1, bc(-e0.z), fma2(up, bc(e1.x), mul2(vp, bc(e1.z)))));
  const float2 ry = fma2(ks, q.dy, fma2(c1, bc(-e0.w), fma2(up, bc(e1.y), mul2(vp, bc(e1.w)))));
  v[LY::nat(0)] = dot2(dnu, bc(q.dx));
  v[LY::nat(1)] = dot2(dnu, q.dy);
  v[LY::nat(2)] = dot2(dnv, bc(q.dx));
  v[LY::nat(3)] = dot2(dnv, q.dy);
  v[LY::nat(4)] = dot2(dden, bc(q.dx));
  v[LY::nat(5)] = dot2(dden, q.dy);
  v[LY::nat(6)] = dot2(nd[0], rx);
  v[LY::nat(7)] = dot2(nd[0], ry);
  v[LY::nat(8)] = hsum(zr2);
  v[LY::nat(9)] = dot2(dzv, rd);
  v[LY::nat(10)] = hsum(nd[0]);
  v[LY::nat(11)] = dot2(w, p.gC[0][0]);
  v[LY::nat(12)] = dot2(w, p.gC[0][1]);
  v[LY::nat(13)] = dot2(w, p.gC[0][2]);
  v[LY::nat(14)] = dot2(nd[1], rx);
  v[LY::nat(15)] = dot2(nd[1], ry);
  v[LY::nat(16)] = dot2(nd[2], rx);
  v[LY::nat(17)] = dot2(nd[2], ry);
  if constexpr (!kLoss) {
    v[LY::nat(18)] = dot2(w, p.gN0);
    v[LY::nat(19)] = dot2(w, p.gN1);
    v[LY::nat(20)] = dot2(w, p.gN2);
  }
}

constexpr float kMinNormal = 1.17549435e-38f;

// The double with the value of a normal, finite v (a conversion instruction
// runs at one warp per 17 clocks of an SM here, measured; these are five
// integer operations).
__device__ __forceinline__ double widen(float v) {
  const uint32_t b = __float_as_uint(v);
  const uint32_t hi = ((uint32_t)((int)b >> 3) & 0x8fffffffu) + 0x38000000u;
  return __hiloint2double((int)hi, (int)(b << 29));
}

// One CTA per tile, one warp per 8 x 8 block.  Each lane group adds its sums
// of an entry straight to the surfel's gradient row in global memory.  That
// leaves the warps without a barrier, an accumulator to clear or a
// compare-and-swap loop (which is what a shared-memory float addition
// compiles to).  The rows are double: there are three to eight times as many
// additions to a row as with one per (surfel, tile), and in float they cost
// accuracy (the scale gradient's error against 64 bits went from 2.3e-5 to
// 4.8e-5 of its norm on a 300k-surfel view).  5.5 million additions of a whole
// row, about what a 1M-surfel view has, take 0.21 ms when nothing else runs
// (0.12 ms in float).
// Rows [lo, lo + rows) of the surfels are present; the other surfels' sums
// are dropped (gs_backward makes several passes when it gets no memory for
// all rows at once).
// Four CTAs per SM (up to 128 registers): with five the code spills (720 ->
// 767 us on the 1M-surfel view, 5.0 -> 5.7 ms for the four backwards of a 4M
// training step).
template <bool kLoss>
__global__ void __launch_bounds__(kThreads, 4) blend_bwd_kernel(
    CamDev cam, SetDev set, const uint32_t* __restrict__ order, const float4* __restrict__ rec,
    const uint16_t* __restrict__ masks, const uint32_t* __restrict__ vals, const int2* __restrict__ ranges,
    const float* __restrict__ out, const int32_t* __restrict__ last, const int32_t* __restrict__ med,
    AdjDev adj, double* __restrict__ grow, uint32_t lo, uint32_t rows, unsigned long long* __restrict__ counters) {
  using LY = Layout<kLoss>;
  constexpr int kN = LY::kN;
  __shared__ WarpSmem sh[kThreads / 32];
  const int tile = order ? (int)order[blockIdx.x] : (int)blockIdx.x;
  const int tx0 = (tile % cam.tiles_x) * kTile, ty0 = (tile / cam.tiles_x) * kTile;
  const int blk = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int lxi = local_x(threadIdx.x), lyi = local_y(threadIdx.x);
  const int px = tx0 + lxi, pyA = ty0 + lyi, pyB = pyA + kRowStep;
  const float lx = (float)lxi + 0.5f;
  const float2 ly = make_float2((float)lyi + 0.5f, (float)(lyi + kRowStep) + 0.5f);
  const int2 rg = ranges[tile];
  const size_t HW = (size_t)cam.W * cam.H;
  const int nsets = adj.n_sets;
  const bool inA = px < cam.W && pyA < cam.H, inB = px < cam.W && pyB < cam.H;
  BwdPix p;
  bwd_init(p, bwd_load<kLoss>(inA, inA ? (size_t)pyA * cam.W + px : 0, HW, out, last, med, adj, set),
           bwd_load<kLoss>(inB, inB ? (size_t)pyB * cam.W + px : 0, HW, out, last, med, adj, set));
  // the lane group's own last blended position: entries behind it are dead for
  // all of its pixels and are not visited
  int glast = max(p.lastA, p.lastB);
#pragma unroll
  for (int o = kGroup / 2; o > 0; o >>= 1) glast = max(glast, __shfl_xor_sync(0xffffffffu, glast, o));
  const int wlast = max(max(__shfl_sync(0xffffffffu, glast, 0), __shfl_sync(0xffffffffu, glast, 8)),
                        max(__shfl_sync(0xffffffffu, glast, 16), __shfl_sync(0xffffffffu, glast, 24)));
  // where the lane's sums go within a row
  const int r = lane & (kGroup - 1);
  double* const dst = grow + r;
  int off1 = -1, off2 = -1;
#pragma unroll
  for (int x = 0; x < kGroup; ++x) {
    if (x == r) {
      off1 = LY::at(x, 1) - x;
      off2 = LY::at(x, 2) - x;
    }
  }
  const bool has1 = off1 + r >= 0, has2 = off2 + r >= 0;
  unsigned replayed = 0, wentries = 0, wlanes = 0;
  WarpSmem& sm = sh[blk];
  walk_list<true>(sm, rec, masks + rg.x, vals + rg.x, 0, wlast, glast, tx0, ty0, blk, 0,
                  [&](int k, int&) {
    const float4 e0 = at16(sm.s0, k), jh = at16(sm.s1, k), e2 = at16(sm.s2, k), jl = at16(sm.s4, k);
    const uint2 meta = at16(sm.meta, k);
    const Pair q = eval_pair(lx, ly, e0, jh, jl, at16(sm.s5, k), e2.y, set);
    const int pos = (int)meta.x;
    const bool liveA = pos < p.lastA, liveB = pos < p.lastB;
    const bool hitA = liveA & q.hitA, hitB = liveB & q.hitB;
    replayed += (liveA ? 1u : 0u) + (liveB ? 1u : 0u);  // performance counter, as wentries and wlanes
    const unsigned ballot = __ballot_sync(0xffffffffu, hitA | hitB);
    if (ballot == 0u) return;
    ++wentries;
    wlanes += __popc(ballot);
    float v[kN];
    // Ji = Jh + Jl (FP32) for the chain rule
    const float4 e1 = make_float4(jh.x + jl.x, jh.y + jl.y, jh.z + jl.z, jh.w + jl.w);
    bwd_pair<kLoss>(p, q, hitA, hitB, e0, e1, e2, at16(sm.s3, k), pos, nsets, set, v);
    rs_level<kGroup / 2, kN>(v, lane);
    const uint32_t row = meta.y - lo;
    if (((ballot >> (lane & 24)) & 0xffu) && row < rows) {
      double* const d = dst + (size_t)row * grad_row_stride(kLoss);
      const float a0 = fabsf(v[0]), a1 = has1 ? fabsf(v[1]) : 0.f, a2 = has2 ? fabsf(v[2]) : 0.f;
      if (a0 + a1 + a2 < INFINITY) {
        // zeros (and what is below the normal range) add nothing
        if (a0 >= kMinNormal) atomicAdd(d, widen(v[0]));
        if (a1 >= kMinNormal) atomicAdd(d + off1, widen(v[1]));
        if (a2 >= kMinNormal) atomicAdd(d + off2, widen(v[2]));
      } else {  // infinities and NaN go through as they are
        atomicAdd(d, (double)v[0]);
        if (has1) atomicAdd(d + off1, (double)v[1]);
        if (has2) atomicAdd(d + off2, (double)v[2]);
      }
    }
  });
  if (counters) {
    unsigned e = replayed;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) e += __shfl_xor_sync(0xffffffffu, e, o);
    if (lane == 0) {
      atomicAdd(&counters[2], (unsigned long long)e);
      atomicAdd(&counters[3], (unsigned long long)wentries);
      atomicAdd(&counters[4], (unsigned long long)wlanes);
    }
  }
}

// ---------------------------------------------------------------------------
// Trim contribution (Sec. 3.3, Eq. 3).
//
// The tiles of the render walk their lists front to back as the forward
// does, with the forward's decisions (same evaluation, same transmittance
// sequence), but every pixel goes through the whole list: a pair that lies
// in the surfel's support (rho <= rho_max) counts towards |P_k| even behind
// the pixel's stop.  A blended pair adds alpha^gamma T^(1 - gamma), T the
// transmittance in front of it.  Per entry a lane group counts its support
// pixels with ballots, sums its contributions with shuffles and adds both to
// the surfel's totals.

__device__ __forceinline__ float contrib_step(float& T, bool& stopped, bool hit, float alpha, const SetDev& set,
                                              float gamma) {
  float c = 0.f;
  if (!stopped && hit) {
    const float Tn = T * (1.f - alpha);
    if (Tn < set.T_min) {
      stopped = true;
    } else {
      c = gamma == 0.5f ? sqrtf(alpha * T) : exp2f(gamma * log2f(alpha) + (1.f - gamma) * log2f(T));
      T = Tn;
    }
  }
  return c;
}

__global__ void __launch_bounds__(kThreads, 5) blend_contrib_kernel(
    CamDev cam, SetDev set, float gamma, const uint32_t* __restrict__ order,
    const float4* __restrict__ rec, const uint16_t* __restrict__ masks, const uint32_t* __restrict__ vals,
    const int2* __restrict__ ranges, float* __restrict__ csum, uint32_t* __restrict__ ccnt) {
  __shared__ WarpSmem sh[kThreads / 32];
  const int tile = order ? (int)order[blockIdx.x] : (int)blockIdx.x;
  const int tx0 = (tile % cam.tiles_x) * kTile, ty0 = (tile / cam.tiles_x) * kTile;
  const int lxi = local_x(threadIdx.x), lyi = local_y(threadIdx.x);
  const int px = tx0 + lxi, pyA = ty0 + lyi, pyB = pyA + kRowStep;
  const int blk = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const float lx = (float)lxi + 0.5f;
  const float2 ly = make_float2((float)lyi + 0.5f, (float)(lyi + kRowStep) + 0.5f);
  const bool inA = px < cam.W && pyA < cam.H, inB = px < cam.W && pyB < cam.H;
  const int2 rg = ranges[tile];
  float TA = 1.f, TB = 1.f;
  bool stA = !inA, stB = !inB;
  WarpSmem& sm = sh[blk];
  walk_list<false>(sm, rec, masks + rg.x, vals + rg.x, 0, rg.y - rg.x, 0, tx0, ty0, blk, 0,
                   [&](int k, int&) {
    const Pair q = eval_pair(lx, ly, at16(sm.s0, k), at16(sm.s1, k), at16(sm.s4, k), at16(sm.s5, k), at16(sm.s2, k).y,
                             set);
    const unsigned ba = __ballot_sync(0xffffffffu, inA & (q.rho.x <= set.rho_max));
    const unsigned bb = __ballot_sync(0xffffffffu, inB & (q.rho.y <= set.rho_max));
    if ((ba | bb) == 0u) return;
    const int sft = lane & 24;
    const uint32_t cnt = (uint32_t)(__popc((ba >> sft) & 0xffu) + __popc((bb >> sft) & 0xffu));
    float c = contrib_step(TA, stA, q.hitA, q.alpha.x, set, gamma) +
              contrib_step(TB, stB, q.hitB, q.alpha.y, set, gamma);
    if (__any_sync(0xffffffffu, c != 0.f)) {
#pragma unroll
      for (int o = kGroup / 2; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
    }
    if (cnt != 0u && (lane & 7) == 0) {
      const uint32_t sid = at16(sm.meta, k).y;
      atomicAdd(&ccnt[sid], cnt);
      if (c != 0.f) atomicAdd(&csum[sid], c);
    }
  });
}

}  // namespace

cudaError_t launch_blend_fwd(const CamDev& cam, const SetDev& set, const uint32_t* order, const float4* rec,
                             const uint16_t* masks, const uint32_t* vals, const int2* ranges, float* out,
                             int32_t* n_contrib, int32_t* last, int32_t* med,
                             unsigned long long* counters, cudaStream_t st) {
  const unsigned grid = (unsigned)cam.tiles_x * (unsigned)cam.tiles_y;
  ProfScope ps(kProfBlendFwd, st);
  // the positions are the backward's; a render that keeps no frame does without
  if (last || med)
    blend_fwd_kernel<true><<<grid, kThreads, 0, st>>>(cam, set, order, rec, masks, vals, ranges, out, n_contrib, last,
                                                      med, counters, 0);
  else
    blend_fwd_kernel<false><<<grid, kThreads, 0, st>>>(cam, set, order, rec, masks, vals, ranges, out, n_contrib, last,
                                                       med, counters, 0);
  count_launch();
  return cudaGetLastError();
}

size_t seg_part_bytes() { return sizeof(SegPart); }

cudaError_t launch_blend_fwd_split(const CamDev& cam, const SetDev& set, const uint32_t* order, const float4* rec,
                                   const uint16_t* masks, const uint32_t* vals, const int2* ranges, float* out,
                                   int32_t* n_contrib, int32_t* last, int32_t* med, unsigned long long* counters,
                                   const SegBufs& sb, cudaStream_t st) {
  const int ntiles = cam.tiles_x * cam.tiles_y;
  ProfScope ps(kProfBlendFwd, st);
  count_launch(2);
  seg_count_kernel<<<div_up(ntiles, 256), 256, 0, st>>>(ranges, ntiles, sb.lseg, sb.segcnt);
  cudaError_t e = launch_scan(sb.segcnt, sb.segoff, ntiles, sb.nseg, sb.scan_tmp, st);
  if (e != cudaSuccess) return e;
  seg_list_kernel<<<div_up(ntiles, 256), 256, 0, st>>>(sb.segcnt, sb.segoff, ntiles, sb.seg_tile, sb.seg_idx);
  // grids sized for the bound, the device count decides
  count_launch(3);
  seg_trans_kernel<<<(unsigned)ntiles + sb.nseg_max, kThreads, 0, st>>>(cam, set, order, rec, masks, vals, ranges, out,
                                                                        n_contrib, last, med, counters, sb.lseg,
                                                                        sb.seg_tile, sb.seg_idx, sb.nseg, sb.trans);
  seg_blend_kernel<<<sb.nseg_max, kThreads, 0, st>>>(cam, set, rec, masks, vals, ranges, sb.lseg, sb.seg_tile,
                                                     sb.seg_idx, sb.nseg, sb.trans,
                                                     static_cast<SegPart*>(sb.part), counters);
  seg_merge_kernel<<<sb.nseg_max, kThreads, 0, st>>>(cam, set, rec, vals, ranges, sb.segcnt, sb.seg_tile,
                                                     sb.seg_idx, sb.nseg, static_cast<const SegPart*>(sb.part),
                                                     out, n_contrib, last, med);
  return cudaGetLastError();
}

cudaError_t launch_blend_fwd_batched(const BlendBatch& batch, int grid, cudaStream_t st) {
  ProfScope ps(kProfBlendFwd, st);
  blend_fwd_batched_kernel<<<grid, kThreads, 0, st>>>(batch);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_blend_bwd(const CamDev& cam, const SetDev& set, const uint32_t* order, const float4* rec,
                             const uint16_t* masks, const uint32_t* vals, const int2* ranges, const float* out,
                             const int32_t* last, const int32_t* med, const AdjDev& adj,
                             bool loss_layout, double* grow, uint32_t lo, uint32_t rows,
                             unsigned long long* counters, cudaStream_t st) {
  const unsigned grid = (unsigned)cam.tiles_x * (unsigned)cam.tiles_y;
  ProfScope ps(kProfBlendBwd, st);
  if (loss_layout)
    blend_bwd_kernel<true><<<grid, kThreads, 0, st>>>(cam, set, order, rec, masks, vals, ranges, out, last, med, adj,
                                                      grow, lo, rows, counters);
  else
    blend_bwd_kernel<false><<<grid, kThreads, 0, st>>>(cam, set, order, rec, masks, vals, ranges, out, last, med, adj,
                                                       grow, lo, rows, counters);
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_blend_contrib(const CamDev& cam, const SetDev& set, float gamma, const uint32_t* order,
                                 const float4* rec, const uint16_t* masks, const uint32_t* vals,
                                 const int2* ranges, float* csum, uint32_t* ccnt, cudaStream_t st) {
  const unsigned grid = (unsigned)cam.tiles_x * (unsigned)cam.tiles_y;
  ProfScope ps(kProfContrib, st);
  blend_contrib_kernel<<<grid, kThreads, 0, st>>>(cam, set, gamma, order, rec, masks, vals, ranges, csum,
                                                  ccnt);
  count_launch();
  return cudaGetLastError();
}

}  // namespace gs2d
