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
// for d L / d alpha.  A warp takes 8 x 8 pixels, two per thread, and the
// entries that reach any of its four 4 x 4 blocks.  A thread adds the
// gradients of its two pixels, the warp reduces them with a reduce-scatter of
// shuffles (one reduction per 64 pixels), the tile sums them in shared memory,
// and they reach global memory once per (surfel, tile).
//
// The order of those FP32 sums is part of the result.  For a long disk seen
// nearly edge-on they cancel, and the gradients of its rotation and size follow
// the rounding of every term and of every partial sum: with other orders of
// the additions, or sums in double, single values moved by up to 2e-3 of the
// gradient's root mean square (seen in a third of the training steps of 4M
// surfels).  So the pairs' terms and the levels of the sum stay as they are,
// although lane groups of eight that walk their own lists and add their sums
// to the surfel's row in double took 768 instead of 1117 us (1M-surfel 1600 x
// 900 view) and 4930 instead of 8430 (the four backwards of the training step).
//
// All are bound by instruction issue, so the time is (group, entry) or (warp,
// entry) steps times instructions per step.  With one list per warp (8 x 8
// pixels) only 10 (4M-surfel orbit view) to 18 (1M aerial view) of a step's 32
// lanes blend anything; 4 x 4 blocks cost a forward warp the longest of its
// four lists instead of their union, and packed FP32 does a thread's two
// pixels in one instruction.  Forward, us (1M-surfel 1600 x 900 view, 4M-surfel
// 1080p view):
//   one list per warp, scalar FP32          501  1148
//   one list per group                      335   690
//   packed FP32                             294   583
//   low part in the rows' order             300   586
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

// Pixels of thread t within its tile (not in the backward): warp w covers columns 8 (w & 1) .. +7
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
// sm holds the entries' block masks (bit 4 w + g).  Returns the length of the
// caller's group's list.
template <int NB>
constexpr int kListStride = NB + 4;  // padded: a walk reads one index past its list
template <int NB>
__device__ __forceinline__ int group_lists(const uint16_t* sm, int nb, int warp, int lane,
                                           uint8_t (*list)[kListStride<NB>]) {
  const uint32_t lt = (1u << lane) - 1u;
  int base[4] = {0, 0, 0, 0};
#pragma unroll
  for (int j = 0; j < NB / 32; ++j) {
    const int e = 32 * j + lane;
    const uint32_t m = e < nb ? (uint32_t)sm[e] >> (4 * warp) : 0u;
#pragma unroll
    for (int g = 0; g < 4; ++g) {
      const bool in = (m >> g) & 1u;
      const uint32_t b = __ballot_sync(0xffffffffu, in);
      if (in) list[g][base[g] + __popc(b & lt)] = (uint8_t)e;
      base[g] += __popc(b);
    }
  }
  __syncwarp();
  const int g = lane >> 3;
  return g == 0 ? base[0] : (g == 1 ? base[1] : (g == 2 ? base[2] : base[3]));
}

// One warp's window on its tile's list (the trim contribution): the entries
// that reach its 8 x 8 block, staged 32 at a time into the two halves of a
// ring, and for each of the warp's four lane groups the ring slots of the
// entries that reach the group's 4 x 4 block, in list order.
constexpr int kHalf = 32;
constexpr int kRing = 2 * kHalf;
constexpr int kQueue = kRing;
struct WarpSmem {
  // slot kRing: an entry that no pixel is near, for the groups whose list is used up
  float4 s0[kRing + 1], s1[kRing + 1], s2[kRing + 1], s4[kRing + 1], s5[kRing + 1];
  uint32_t sid[kRing + 1];  // surfel
  uint32_t q[kQueue];       // surfels found but not yet staged (a ring)
  uint8_t qm[kQueue];       // and their group masks
  uint16_t list[4][kRing];  // per group, byte offsets of ring slots (16 x slot; a ring of its own)
};
// Element of a staged array at a byte offset that is 16 times its slot.
__device__ __forceinline__ float4 at16(const float4* a, int k) {
  return *reinterpret_cast<const float4*>(reinterpret_cast<const char*>(a) + k);
}

// Walks the len entries of a tile's list front to back for one warp (its block
// blk).  body(k) is called with every lane: k is the offset (16 x ring slot) of
// the lane's group's next entry; a group whose list is used up for now gets an
// entry that misses every pixel.
//
// The warps of a CTA share no data and no barrier: with one staging per CTA
// and batch, a quarter of the warps' time went to waiting for the slowest
// warp and for the staging loads.  A group may run ahead of the others by
// up to one half of the ring, which evens out most of the difference between
// the groups' lists (the older half is refilled when all groups are past it).
template <class Body>
__device__ __forceinline__ void walk_list(WarpSmem& sm, const float4* __restrict__ rec,
                                          const uint16_t* __restrict__ masks, const uint32_t* __restrict__ vals,
                                          int len, int tx0, int ty0, int blk, Body body) {
  constexpr unsigned kFull = 0xffffffffu;
  const int lane = threadIdx.x & 31, g = lane >> 3;
  const uint32_t lt = (1u << lane) - 1u;
  int scan = 0, qn = 0, q0 = 0;
  uint32_t pm = 0u, pv = 0u;  // the next 32 entries' masks and surfels, loaded ahead
  auto load = [&] {
    const int e = scan + lane;
    pm = e < len ? masks[e] : 0u;
    pv = e < len ? vals[e] : 0u;
  };
  load();
  if (lane == 0) {
    sm.s0[kRing] = make_float4(1e15f, 1e15f, 0.f, 0.f);
    sm.s1[kRing] = sm.s4[kRing] = make_float4(0.f, 0.f, 0.f, 0.f);
    sm.s2[kRing] = make_float4(1.f, 0.f, 0.f, 0.f);
    sm.s5[kRing] = make_float4(__int_as_float(0x7fffffff), 0.f, 0.f, 0.f);
    sm.sid[kRing] = 0u;
  }
  // entries staged so far for the lane's group, those of them it has walked, and
  // for all four groups the staged ones modulo the ring (one byte each)
  int end = 0, i = 0, h = 0;
  uint32_t cnt = 0u;
  for (;;) {
    int mid = end;  // the older half's
    const bool fill = qn > 0 || scan < len;
    if (fill) {
      __syncwarp();  // every lane is done with the older half
      while (qn < kHalf && scan < len) {
        const uint32_t m = (pm >> (4 * blk)) & 15u, v = pv;
        scan += 32;
        if (scan < len) load();
        const uint32_t b = __ballot_sync(kFull, m != 0u);
        if (m != 0u) {
          const int slot = (q0 + qn + __popc(b & lt)) & (kQueue - 1);
          sm.q[slot] = v;
          sm.qm[slot] = (uint8_t)m;
        }
        qn += __popc(b);
      }
      __syncwarp();
      const int nb = min(qn, kHalf);
      const int slot = h * kHalf + lane;
      uint32_t m = 0u;
      if (lane < nb) {
        const uint32_t v = sm.q[(q0 + lane) & (kQueue - 1)];
        m = sm.qm[(q0 + lane) & (kQueue - 1)];
        const Staged e = stage_entry(rec, v, tx0, ty0);
        sm.s0[slot] = e.s0;
        sm.s1[slot] = e.s1;
        sm.s2[slot] = e.s2;
        sm.s4[slot] = e.s4;
        sm.s5[slot] = e.s5;
        sm.sid[slot] = v;
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
      body(k);
    }
    if (!fill) break;
  }
}

// One entry against a thread's two pixels A and B (one column, kRowStep rows
// apart); the halves of each pair are the two pixels.
struct Pair {
  float dx;        // pixel offset from the projected centre (the column is shared)
  float2 dy;
  float2 nu, nv;   // Ji d
  float2 rden;     // 1 / (1 + e.d)
  float2 rho;      // min(rho_obj, rho_scr)
  float2 G;        // exp(-rho / 2)
  float2 alpha;    // min(alpha_max, o G)
  bool objA, objB; // object-space branch
  bool hitA, hitB; // rho <= rho_max and alpha >= alpha_min
};

// The exact grid sums nu0h + Jh (lx, ly) plus the small low-part corrections
// (see Staged), then the ray-splat distance, the screen filter and alpha.
// Shared by every blend; explicit round-to-nearest operations so that
// the forward and the backward take bit-identical decisions.  The rows are
// lb + off: lb the row four above where the pixel lies in the lower half of its
// 8 x 8 block (off 4), else its own (off 0).  The low part reaches a lower row
// by a step of 4 Jl from the upper one, in every blend.
__device__ __forceinline__ Pair eval_pair(float lx, float2 lb, float2 off, float4 s0, float4 jh, float4 jl, float4 n0,
                                          float opac, const SetDev& set) {
  Pair q;
  const float2 ly = add2(lb, off);
  const float su = __fmaf_rn(jh.x, lx, n0.x), sv = __fmaf_rn(jh.z, lx, n0.y);  // exact, the column's part
  const float2 cu = fma2(bc(jl.y), off, fma2(bc(jl.x), bc(lx), fma2(bc(jl.y), lb, bc(n0.z))));
  const float2 cv = fma2(bc(jl.w), off, fma2(bc(jl.z), bc(lx), fma2(bc(jl.w), lb, bc(n0.w))));
  q.nu = add2(fma2(bc(jh.y), ly, bc(su)), cu);
  q.nv = add2(fma2(bc(jh.w), ly, bc(sv)), cv);
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
  q.G = make_float2(ex2_approx(x.x), ex2_approx(x.y));
  const float2 a = mul2(bc(opac), q.G);
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
                                         float2 lb, float2 off, const SetDev& set) {
  if (p.doneA && p.doneB) return;
  int k = list[0];
  for (int i = 0; i < glen; ++i) {
    const float4 e0 = sh.s0[k], e1 = sh.s1[k], e2 = sh.s2[k], e3 = sh.s3[k], e4 = sh.s4[k], e5 = sh.s5[k];
    const int pos = b0 + k;
    k = list[i + 1];  // past the end: a byte of padding, not used
    const Pair q = eval_pair(lx, lb, off, e0, e1, e4, e5, e2.y, set);
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
  const float2 off = bc((float)(lyi & 4));
  const float2 lb = make_float2((float)(lyi & ~4) + 0.5f, (float)((lyi & ~4) + kRowStep) + 0.5f);
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
    fwd_walk<false, kPos>(p, sh, sh.list[warp][lane >> 3], glen, b0, lx, lb, off, set);
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
  const float2 off = bc((float)(lyi & 4));
  const float2 lb = make_float2((float)(lyi & ~4) + 0.5f, (float)((lyi & ~4) + kRowStep) + 0.5f);
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
      const Pair q = eval_pair(lx, lb, off, sh.s0[k], sh.s1[k], sh.s4[k], sh.s5[k], sh.s2[k].y, set);
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
  const float2 off = bc((float)(lyi & 4));
  const float2 lb = make_float2((float)(lyi & ~4) + 0.5f, (float)((lyi & ~4) + kRowStep) + 0.5f);
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
    fwd_walk<true, true>(p, sh, sh.list[warp][lane >> 3], glen, b0, lx, lb, off, set);
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
// Entries staged per batch in the backward, by the CTAs per SM its variant
// is sized for: 128 for five (a small batch leaves more of the SM's shared
// memory to L1: 0.939 -> 0.921 ms on the 1M-surfel view, against 224), 224
// for four (the dense variant's long lists: 128 made the 4M-surfel training
// step 2.5 % slower).  The gradient accumulators and the six staged vectors
// per entry fit either way.
constexpr int batch_b(int min_ctas) { return min_ctas >= 5 ? 128 : 224; }
// Average tile-list length from which the backward takes the 4-CTA variant:
// 200 (the 1M-surfel aerial view) ran best with 5 CTAs per SM, 590 (the
// 4M-surfel orbit view) with 4.
constexpr int kDenseListLen = 400;

// Per-pair gradient vector.  General layout (any adjoint planes):
//   [0..5] d Ji, d e; [6] Zc, the depth term of the centre gradient (below);
//   [7] d p_z, [8] d opacity, [9..11] d rgb, [12..14] d normal;
//   [15 + 2 s, 16 + 2 s] screen-space gradient of set s.
// Loss layout (set 0 on colour and inverse depth only, later sets on
// colour): the normal slots are dropped, [0..11] as above without d normal,
// [12 + 2 s, 13 + 2 s] screen gradients.
// The centre gradient is not accumulated on its own: per pair it is set 0's
// screen gradient plus, on the object-space branch, the term of the depth
// z = p_z / (1 + e.d) through d, (d rden / d d) p_z dz = -e p_z rden^2 dz;
// so d c = (screen gradient of set 0) + e * Zc with Zc the sum of
// p_z rden^2 dz, formed once per entry at the flush.
template <bool kLoss>
struct Layout {
  static constexpr int kRec = kLoss ? 12 : kGradRec - 1;
  static constexpr int kN = kRec + 2 * kMaxSets;  // 18 or 21
};

// Balanced reduce-scatter of N values over the warp: at each halving level
// the lanes whose bit is clear keep the first ceil(N/2) values and the others
// the rest, exchanging the halves they do not keep; N values need about
// N + 5 shuffles.  Afterwards v[0] holds the warp sum of one slot, given by
// rs_slot() for the lane (or nothing when rs_slot() returns -1).
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

template <int N>
__device__ __forceinline__ int rs_slot(int lane) {
  int n = N, real = N, slot = 0;
  for (int o = 16; o >= 1; o >>= 1) {
    const int L = (n + 1) / 2;
    if (lane & o) {
      slot += L;
      real = real - L > 0 ? real - L : 0;
    } else {
      real = real < L ? real : L;
    }
    n = L;
  }
  return real > 0 ? slot : -1;
}

// Pixels of thread t: lane l takes column l & 7 and rows l >> 3 and
// (l >> 3) + kBwdRowStep of its warp's 8 x 8 block.
constexpr int kBwdRowStep = 4;
__device__ __forceinline__ int bwd_x(int t) { return (((t >> 5) & 1) << 3) | (t & 7); }
__device__ __forceinline__ int bwd_y(int t) { return ((t >> 6) << 3) | ((t >> 3) & 3); }

// Per warp, the batch's entries that reach any of the warp's four 4 x 4 blocks
// (bits 4 w .. 4 w + 3 of the block masks), as NW bit words; the loops below
// visit only their set bits.
template <int NW>
__device__ __forceinline__ void warp_entry_bits(const uint16_t* sm, int nb, int warp, int lane, uint32_t* wb) {
#pragma unroll
  for (int j = 0; j < NW; ++j) {
    const int e = 32 * j + lane;
    const uint32_t w = __ballot_sync(0xffffffffu, e < nb && ((sm[e] >> (4 * warp)) & 15u));
    if (lane == 0) wb[j] = w;
  }
  __syncwarp();
}

// One pixel's half of a Pair.
struct PixPair {
  float dx, dy, nu, nv, rden, rho, G, alpha;
  bool obj, hit;
};
__device__ __forceinline__ PixPair pair_a(const Pair& q) {
  return {q.dx, q.dy.x, q.nu.x, q.nv.x, q.rden.x, q.rho.x, q.G.x, q.alpha.x, q.objA, q.hitA};
}
__device__ __forceinline__ PixPair pair_b(const Pair& q) {
  return {q.dx, q.dy.y, q.nu.y, q.nv.y, q.rden.y, q.rho.y, q.G.y, q.alpha.y, q.objB, q.hitB};
}

// Per-pixel state of the reverse replay: transmittance, suffix sums S of
// each adjoint set, the pixel's adjoints, and (general layout) the running
// opacity A and depth sum Z with their final values for the distortion.
struct BwdPix {
  float T, A, Z, Af, Zf;
  float S[kMaxSets];
  float gC[kMaxSets][3];
  float gA, gZ, gI, gMed, gD, gN0, gN1, gN2;
  int last, med;
};

template <bool kLoss>
__device__ __forceinline__ void bwd_init(BwdPix& p, bool inside, size_t pix, size_t HW,
                                         const float* __restrict__ out, const int32_t* __restrict__ last,
                                         const int32_t* __restrict__ med, const AdjDev& adj,
                                         const SetDev& set) {
  p.T = 1.f;
  p.A = p.Z = p.Af = p.Zf = 0.f;
  p.gA = p.gZ = p.gI = p.gMed = p.gD = p.gN0 = p.gN1 = p.gN2 = 0.f;
  p.last = 0;
  p.med = -1;
#pragma unroll
  for (int s = 0; s < kMaxSets; ++s) {
    p.gC[s][0] = p.gC[s][1] = p.gC[s][2] = 0.f;
    p.S[s] = 0.f;
  }
  if (!inside) return;
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
    p.Af = p.A = out[3 * HW + pix];
    p.Zf = p.Z = out[4 * HW + pix];
    if (m & (1u << 3)) p.gA = a[3 * HW + pix];
    if (m & (1u << 4)) p.gZ = a[4 * HW + pix];
    if (m & (1u << 6)) p.gMed = a[6 * HW + pix];
    if (m & (1u << 7)) p.gN0 = a[7 * HW + pix];
    if (m & (1u << 8)) p.gN1 = a[8 * HW + pix];
    if (m & (1u << 9)) p.gN2 = a[9 * HW + pix];
    if (m & (1u << 10)) p.gD = a[10 * HW + pix];
  }
}

// A pair that was not blended (or lies past the pixel's last blended
// entry) is masked so that every term of bwd_pair is a finite zero and the
// pixel's state passes through unchanged: alpha = G = 0 and the
// screen-space branch, whose terms are finite for any offset.
__device__ __forceinline__ void mask_pair(PixPair& q, bool live) {
  const bool h = live && q.hit;
  q.hit = h;
  q.alpha = h ? q.alpha : 0.f;
  q.G = h ? q.G : 0.f;
  q.obj = h && q.obj;
}

// Gradient of one pair at list position k, added into v (gradient-vector
// layout), and the pixel's replay state moved past it.  Branch-free, so that
// the two pixels of a thread interleave: both branches of the ray-splat are
// formed and the one the forward took is selected.
template <bool kLoss>
__device__ __forceinline__ void bwd_pair(BwdPix& p, const PixPair& q, float4 e0, float4 e1, float4 e2,
                                         float4 e3, int k, int nsets, const SetDev& set, float* v) {
  using LY = Layout<kLoss>;
  const float rom = rcp_approx(1.f - q.alpha);
  p.T = q.hit ? p.T * rom : p.T;  // transmittance before this pair
  const float w = q.alpha * p.T;
  const float pz = e2.x;
  const float z = q.obj ? pz * q.rden : pz;
  const float rz = rcp_approx(z);
  float dLdw = p.gC[0][0] * e2.z + p.gC[0][1] * e2.w + p.gC[0][2] * e3.x + p.gI * rz;
  float dzv = -w * p.gI * rz * rz;
  if constexpr (!kLoss) {
    const float Ap = p.A - w, Zp = p.Z - w * z;
    const float dDdw = 2.f * (z * Ap - Zp + (p.Zf - p.Z) - z * (p.Af - p.A));
    dLdw += p.gA + p.gZ * z + p.gN0 * e3.y + p.gN1 * e3.z + p.gN2 * e3.w + p.gD * dDdw;
    dzv += w * p.gZ + p.gD * 2.f * w * (Ap - (p.Af - p.A)) + (k == p.med ? p.gMed : 0.f);
    p.A = Ap;
    p.Z = Zp;
  }
  float dLda[kMaxSets];
  dLda[0] = p.T * dLdw - p.S[0] * rom;
  p.S[0] += w * dLdw;
#pragma unroll
  for (int s = 1; s < kMaxSets; ++s) {
    if (s < nsets) {
      const float dw = p.gC[s][0] * e2.z + p.gC[s][1] * e2.w + p.gC[s][2] * e3.x;
      dLda[s] = p.T * dw - p.S[s] * rom;
      p.S[s] += w * dw;
    } else {
      dLda[s] = 0.f;
    }
  }
  // alpha -> rho (zero where alpha is clamped at alpha_max).  Every
  // derivative of rho below carries a factor 2; it is kept in
  // dadrho2 = 2 d alpha / d rho and drho2 = 2 dL / d rho (exact scalings),
  // and rx, ry are half of d rho / d d.
  const bool unclamped = e2.y * q.G < set.alpha_max;
  const float dadrho2 = unclamped ? -q.alpha : 0.f;
  const float drho2 = dLda[0] * dadrho2;
  // object-space branch: rho = u^2 + v^2 with (u, v) = (nu, nv) rden,
  // z = p_z rden (its terms may be non-finite where it was not taken)
  const float r2d = q.rden * q.rden;
  const float tx = q.nu * e1.x + q.nv * e1.z, ty = q.nu * e1.y + q.nv * e1.w;
  const float c1 = q.rho * q.rden;
  const float u = q.nu * q.rden, vv = q.nv * q.rden;
  const float dnu = u * q.rden * drho2, dnv = vv * q.rden * drho2;
  const float zr2 = dzv * pz * r2d;
  const float drden = drho2 * (u * q.nu + vv * q.nv) + dzv * pz;
  const float dden = -drden * r2d;
  const bool ob = q.obj;
  const float rx = ob ? r2d * tx - c1 * e0.z : set.sinv * q.dx;
  const float ry = ob ? r2d * ty - c1 * e0.w : set.sinv * q.dy;
  const float gpz = ob ? dzv * q.rden : dzv;
  // the object-space terms of Ji, e and the centre's depth term, zero (and
  // finite) where the screen branch was taken
  const float dnu_o = ob ? dnu : 0.f, dnv_o = ob ? dnv : 0.f, dden_o = ob ? dden : 0.f;
  v[0] = fmaf(dnu_o, q.dx, v[0]);
  v[1] = fmaf(dnu_o, q.dy, v[1]);
  v[2] = fmaf(dnv_o, q.dx, v[2]);
  v[3] = fmaf(dnv_o, q.dy, v[3]);
  v[4] = fmaf(dden_o, q.dx, v[4]);
  v[5] = fmaf(dden_o, q.dy, v[5]);
  v[6] += ob ? zr2 : 0.f;
  v[7] += gpz;
  v[8] = fmaf(dLda[0], unclamped ? q.G : 0.f, v[8]);
  v[9] += w * p.gC[0][0];
  v[10] += w * p.gC[0][1];
  v[11] += w * p.gC[0][2];
  if constexpr (!kLoss) {
    v[12] += w * p.gN0;
    v[13] += w * p.gN1;
    v[14] += w * p.gN2;
  }
#pragma unroll
  for (int s = 0; s < kMaxSets; ++s) {
    const float dr = dLda[s] * dadrho2;
    v[LY::kRec + 2 * s] -= dr * rx;
    v[LY::kRec + 2 * s + 1] -= dr * ry;
  }
}

// Shared-memory staging of the backward (one batch of kBB entries).
template <int kAcc, int kBB>
struct BwdSmem {
  float4 s0[kBB], s1[kBB], s2[kBB], s3[kBB], s4[kBB], s5[kBB];
  uint16_t sm[kBB];
  uint32_t sid[kBB];
  float acc[kBB][kAcc];
  uint32_t wbits[kThreads / 32][kBB / 32];
  int smax;
};

// Reverse replay of entry kk (list position k) for a thread's two pixels:
// the pair's gradients, reduced over the warp into the entry's accumulator.
template <bool kLoss, int kN, int kAcc, int kBB>
__device__ __forceinline__ void bwd_entry(BwdSmem<kAcc, kBB>& sh, int kk, int k, float lx, float ly, BwdPix& a,
                                          BwdPix& b, int nsets, const SetDev& set, int lane, int myslot,
                                          unsigned& wentries, unsigned& wlanes) {
  const float4 e0 = sh.s0[kk], jh = sh.s1[kk], e2 = sh.s2[kk];
  const bool liveA = k < a.last, liveB = k < b.last;
  const float4 jl = sh.s4[kk];
  const Pair q = eval_pair(lx, bc(ly), make_float2(0.f, (float)kBwdRowStep), e0, jh, jl, sh.s5[kk], e2.y, set);
  PixPair qa = pair_a(q), qb = pair_b(q);
  mask_pair(qa, liveA);
  mask_pair(qb, liveB);
  const bool contrib = qa.hit || qb.hit;
  const unsigned ballot = __ballot_sync(0xffffffffu, contrib);
  if (ballot == 0u) return;
  ++wentries;
  wlanes += __popc(ballot);
  float v[kN];
#pragma unroll
  for (int i = 0; i < kN; ++i) v[i] = 0.f;
  const float4 e3 = sh.s3[kk];
  // Ji = Jh + Jl (FP32) for the chain rule
  const float4 e1 = make_float4(jh.x + jl.x, jh.y + jl.y, jh.z + jl.z, jh.w + jl.w);
  // a pixel row with no hit in the whole warp needs no gradient pass (a
  // masked pair leaves the pixel's state and the sums unchanged)
  const bool anyA = __any_sync(0xffffffffu, qa.hit), anyB = __any_sync(0xffffffffu, qb.hit);
  if (anyA && anyB) {
    bwd_pair<kLoss>(a, qa, e0, e1, e2, e3, k, nsets, set, v);
    bwd_pair<kLoss>(b, qb, e0, e1, e2, e3, k, nsets, set, v);
  } else if (anyA) {
    bwd_pair<kLoss>(a, qa, e0, e1, e2, e3, k, nsets, set, v);
  } else {
    bwd_pair<kLoss>(b, qb, e0, e1, e2, e3, k, nsets, set, v);
  }
  if (__popc(ballot) == 1) {
    if (contrib) {
#pragma unroll
      for (int i = 0; i < kN; ++i)
        if (v[i] != 0.f) atomicAdd(&sh.acc[kk][i], v[i]);
    }
  } else {
    rs_level<16, kN>(v, lane);
    if (myslot >= 0 && v[0] != 0.f) atomicAdd(&sh.acc[kk][myslot], v[0]);
  }
}

// Records of the surfels [lo, lo + rows) are present; the other surfels' sums
// are dropped (gs_backward makes several passes when it gets no memory for
// all records at once).
// kMinCtas: the CTAs per SM the register budget is sized for (5: 96
// registers; 4: up to 128, for dense lists of small footprints).
template <bool kLoss, int kMinCtas>
__global__ void __launch_bounds__(kThreads, kMinCtas) blend_bwd_kernel(
    CamDev cam, SetDev set, const uint32_t* __restrict__ order, const float4* __restrict__ rec,
    const uint16_t* __restrict__ masks, const uint32_t* __restrict__ vals, const int2* __restrict__ ranges,
    const float* __restrict__ out, const int32_t* __restrict__ last, const int32_t* __restrict__ med,
    AdjDev adj, float* __restrict__ grec, float* __restrict__ screen, int n, uint32_t lo, uint32_t rows,
    unsigned long long* __restrict__ counters) {
  using LY = Layout<kLoss>;
  constexpr int kN = LY::kN;
  constexpr int kAcc = kN | 1;  // odd row stride: the flush's column reads are conflict-free
  constexpr int kBatchB = batch_b(kMinCtas), kWordsB = kBatchB / 32;
  __shared__ BwdSmem<kAcc, kBatchB> sh;
  const int tile = order ? (int)order[blockIdx.x] : (int)blockIdx.x;
  const int tx0 = (tile % cam.tiles_x) * kTile, ty0 = (tile / cam.tiles_x) * kTile;
  const int lxi = bwd_x(threadIdx.x), lyi = bwd_y(threadIdx.x);
  const int px = tx0 + lxi, pyA = ty0 + lyi, pyB = pyA + kBwdRowStep;
  const int warp = threadIdx.x >> 5;
  const float lx = (float)lxi + 0.5f, lyA = (float)lyi + 0.5f;
  const int2 rg = ranges[tile];
  const size_t HW = (size_t)cam.W * cam.H;
  const int lane = threadIdx.x & 31;
  const int nsets = adj.n_sets;
  const int myslot = rs_slot<kN>(lane);
  const bool inA = px < cam.W && pyA < cam.H, inB = px < cam.W && pyB < cam.H;
  BwdPix a, b;
  bwd_init<kLoss>(a, inA, inA ? (size_t)pyA * cam.W + px : 0, HW, out, last, med, adj, set);
  bwd_init<kLoss>(b, inB, inB ? (size_t)pyB * cam.W + px : 0, HW, out, last, med, adj, set);
  if (threadIdx.x == 0) sh.smax = 0;
  __syncthreads();
  atomicMax(&sh.smax, max(a.last, b.last));
  __syncthreads();
  const int maxlast = sh.smax;
  // the warp's own last blended position: entries behind it are dead for all
  // of its pixels and are not visited
  int wlast = max(a.last, b.last);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) wlast = max(wlast, __shfl_xor_sync(0xffffffffu, wlast, o));
  unsigned replayed = 0, wentries = 0, wlanes = 0;

  for (int bend = maxlast; bend > 0; bend -= kBatchB) {
    const int b0 = bend > kBatchB ? bend - kBatchB : 0;
    const int nb = bend - b0;
    __syncthreads();
    for (int t = threadIdx.x; t < nb; t += kThreads) {
      const uint32_t s = vals[rg.x + b0 + t];
      sh.sid[t] = s;
      const Staged e = stage_entry(rec, s, tx0, ty0);
      sh.s0[t] = e.s0;
      sh.s1[t] = e.s1;
      sh.s2[t] = e.s2;
      sh.s3[t] = e.s3;
      sh.s4[t] = e.s4;
      sh.s5[t] = e.s5;
      sh.sm[t] = masks[rg.x + b0 + t];
    }
    for (int i = threadIdx.x; i < nb * kAcc; i += kThreads) (&sh.acc[0][0])[i] = 0.f;
    __syncthreads();
    warp_entry_bits<kWordsB>(sh.sm, nb, warp, lane, sh.wbits[warp]);
    if (lane == 0) {
#pragma unroll
      for (int j = 0; j < kWordsB; ++j) {
        const int lw = wlast - b0 - 32 * j;
        sh.wbits[warp][j] &= lw >= 32 ? 0xffffffffu : (lw > 0 ? (1u << lw) - 1u : 0u);
      }
    }
    __syncwarp();
    if (counters) {
      // the batch's entries before each pixel's last blended one that the
      // warp visits (performance counter)
#pragma unroll
      for (int j = 0; j < kWordsB; ++j) {
        const uint32_t bits = sh.wbits[warp][j];
        const int la = a.last - b0 - 32 * j, lb = b.last - b0 - 32 * j;
        replayed += (unsigned)__popc(la >= 32 ? bits : (la > 0 ? bits & ((1u << la) - 1u) : 0u));
        replayed += (unsigned)__popc(lb >= 32 ? bits : (lb > 0 ? bits & ((1u << lb) - 1u) : 0u));
      }
    }
    for (int j = kWordsB - 1; j >= 0; --j) {
      uint32_t bits = sh.wbits[warp][j];
      while (bits != 0u) {  // back to front: highest set bit first
        const int hb = 31 - __clz(bits);
        bits &= ~(1u << hb);
        bwd_entry<kLoss, kN, kAcc, kBatchB>(sh, 32 * j + hb, b0 + 32 * j + hb, lx, lyA, a, b, nsets, set, lane, myslot,
                                   wentries, wlanes);
      }
    }
    __syncthreads();
    // flush this batch: one (surfel, tile) gradient record per entry, the
    // centre gradient formed from set 0's screen gradient and Zc
    for (int t = threadIdx.x; t < nb; t += kThreads) {
      const uint32_t s = sh.sid[t];
      if (s - lo >= rows) continue;
      float* g = grec + (size_t)(s - lo) * kGradRec;
      const float* x = sh.acc[t];
      const float4 e0 = sh.s0[t];
      float r[kGradRec];
#pragma unroll
      for (int i = 0; i < 6; ++i) r[i] = x[i];
      r[6] = fmaf(e0.z, x[6], x[LY::kRec]);
      r[7] = fmaf(e0.w, x[6], x[LY::kRec + 1]);
#pragma unroll
      for (int i = 7; i < LY::kRec; ++i) r[i + 1] = x[i];
#pragma unroll
      for (int i = 0; i < LY::kRec + 1; ++i)
        if (r[i] != 0.f) atomicAdd(&g[i], r[i]);
      if (screen) {
        for (int st = 0; st < nsets; ++st) {
          const float x0 = sh.acc[t][LY::kRec + 2 * st];
          const float x1 = sh.acc[t][LY::kRec + 2 * st + 1];
          float* sg = screen + ((size_t)st * n + s) * 2;
          if (x0 != 0.f) atomicAdd(&sg[0], x0);
          if (x1 != 0.f) atomicAdd(&sg[1], x1);
        }
      }
    }
  }
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
// the surfel's totals.  A wide, faint surfel gets an addition from every 4 x 4
// block of the image, half a million at 4K: in FP32 each would round the same
// way (an error of a percent there), so the sum is double.

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
    const int2* __restrict__ ranges, double* __restrict__ csum, uint32_t* __restrict__ ccnt) {
  __shared__ WarpSmem sh[kThreads / 32];
  const int tile = order ? (int)order[blockIdx.x] : (int)blockIdx.x;
  const int tx0 = (tile % cam.tiles_x) * kTile, ty0 = (tile / cam.tiles_x) * kTile;
  const int lxi = local_x(threadIdx.x), lyi = local_y(threadIdx.x);
  const int px = tx0 + lxi, pyA = ty0 + lyi, pyB = pyA + kRowStep;
  const int blk = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const float lx = (float)lxi + 0.5f;
  const float2 off = bc((float)(lyi & 4));
  const float2 lb = make_float2((float)(lyi & ~4) + 0.5f, (float)((lyi & ~4) + kRowStep) + 0.5f);
  const bool inA = px < cam.W && pyA < cam.H, inB = px < cam.W && pyB < cam.H;
  const int2 rg = ranges[tile];
  float TA = 1.f, TB = 1.f;
  bool stA = !inA, stB = !inB;
  WarpSmem& sm = sh[blk];
  walk_list(sm, rec, masks + rg.x, vals + rg.x, rg.y - rg.x, tx0, ty0, blk, [&](int k) {
    const Pair q = eval_pair(lx, lb, off, at16(sm.s0, k), at16(sm.s1, k), at16(sm.s4, k), at16(sm.s5, k), at16(sm.s2, k).y,
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
      for (int o = 4; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
    }
    if (cnt != 0u && (lane & 7) == 0) {
      const uint32_t sid = sm.sid[k / 16];
      atomicAdd(&ccnt[sid], cnt);
      if (c != 0.f) atomicAdd(&csum[sid], (double)c);
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
                             const int32_t* last, const int32_t* med, const AdjDev& adj, float* grec, uint32_t lo,
                             uint32_t rows, float* screen, int n, int64_t K, unsigned long long* counters, cudaStream_t st) {
  const unsigned grid = (unsigned)cam.tiles_x * (unsigned)cam.tiles_y;
  // the training loss drives set 0 through colour and inverse depth only and
  // the other sets through colour: a leaner kernel for that layout
  bool loss_layout = (adj.mask[0] & ~(GS_MASK_RGB | (1u << GS_PLANE_INVDEPTH))) == 0u;
  for (int s = 1; s < adj.n_sets; ++s) loss_layout = loss_layout && (adj.mask[s] & ~GS_MASK_RGB) == 0u;
  ProfScope ps(kProfBlendBwd, st);
  const bool dense = K >= (int64_t)kDenseListLen * (int64_t)grid;
#define GS_BWD(L, M)                                                                                           \
  blend_bwd_kernel<L, M><<<grid, kThreads, 0, st>>>(cam, set, order, rec, masks, vals, ranges, out, last, med, \
                                                    adj, grec, screen, n, lo, rows, counters)
  if (loss_layout) {
    if (dense) GS_BWD(true, 4);
    else GS_BWD(true, 5);
  } else {
    if (dense) GS_BWD(false, 4);
    else GS_BWD(false, 5);
  }
#undef GS_BWD
  count_launch();
  return cudaGetLastError();
}

cudaError_t launch_blend_contrib(const CamDev& cam, const SetDev& set, float gamma, const uint32_t* order,
                                 const float4* rec, const uint16_t* masks, const uint32_t* vals,
                                 const int2* ranges, double* csum, uint32_t* ccnt, cudaStream_t st) {
  const unsigned grid = (unsigned)cam.tiles_x * (unsigned)cam.tiles_y;
  ProfScope ps(kProfContrib, st);
  blend_contrib_kernel<<<grid, kThreads, 0, st>>>(cam, set, gamma, order, rec, masks, vals, ranges, csum,
                                                  ccnt);
  count_launch();
  return cudaGetLastError();
}

}  // namespace gs2d
