// The list kernel: pair-distance histograms of spatially ordered species, one
// warp per run of kRun i particles (sm_103a).
//
// Every particle image that can lie in the current bin sweep as seen from the
// run's bounding box is listed once, and every listed image is evaluated
// against the whole run with the same arithmetic whatever the box: no nearest
// image is searched per pair.  With r_max at most half the smallest distance
// between a particle's images, one image of a pair at most lies inside r_max,
// and the others are counted as out of range like any other far pair (those
// whose float32 value comes close to a bin edge are re-decided, and counted
// only for the image that the binary64 definition picks).  So the periodic
// frames cost what the frame without a box costs, and particles beyond r_max
// of the run are dropped one by one, not in tiles.
//
// Per pair of float32 lanes: three FMAs and one add give q = t^2 (the run's
// centre is the origin, so q = |y|^2 + (|x|^2 - 2 x.y) with |y|^2 listed and
// the parenthesis small), then one square root, two adds and one FMA for the
// residual, and the counting step of the tiled kernel.  The paper's kernels
// (Sec. 3.2) evaluate every pair and wrap it per axis (Eq. 5).
//
// Warps claim items of one segment (species pair and sweep) straight from its
// counter; the warps of a block meet only when a segment is exhausted, to merge
// their shared histogram.  Large segments are shared by blocks, small ones are one
// block's own, handed out from one counter: with every block free to choose among all
// segments, those of equal frames were started one after another (10,000 frames of 200
// particles, three species: pair kernel 808 -> 4.2 ms, 2,000 of 2,000: 59 -> 4.1 ms).
//
// What bounds it: without a box the shared-memory pipe (one increment per pair at
// 3.5 wavefronts on random banks, 90 % busy at N = 200,000), for periodic frames
// the issue slots (15 instructions per pair and lane, 70 % of the slots used).
// Pair kernel at 2,070 MHz, 10,000 bins, the tiled kernel before -> now:
// N = 1,000,000 none 235 -> 229 ms, orthorhombic 254 -> 162, triclinic 284 -> 125;
// N = 100,000 orthorhombic, two species 4.2 -> 2.6 ms; N = 500,000 clustered
// triclinic, three species, 20,000 bins 92.6 -> 43 ms; N = 2,000 none, 1,000 bins
// 118 -> 18 us (items small enough for one per warp).
// Measured and not kept: three 256-thread blocks of 80 registers (none 13.2 ms at
// N = 200,000 against 9.6: spills, and the run's factors loaded again per block of
// images), 384 and 448 threads (10.6 and 10.0 ms), sixteen pairs per lane and turn
// instead of thirty-two (10.1 ms).
#include <math.h>
#include <stdint.h>

#include <algorithm>

#include "dh_device.h"
#include "dh_internal.h"

namespace dh {

namespace {

// Listed images evaluated at a time; with 32, two thirds of the lists' shared memory
// for 7,168 bins more (launch_list)
constexpr int kBlk = 64, kBlkNarrow = 32;
constexpr int kImgShift = 26;  // list reference: particle | image << 26
constexpr int kHome = 13;      // the image k = 0
constexpr int kPickCap = 64;   // images evaluated at a time in pick_round (at least 27)
constexpr uint32_t kLastImage = 0x80000000u;
constexpr uint32_t kAnyImage = 31u << kImgShift;  // reference of a pair whose image is chosen by the drain
// A claim takes 1/kClaims of a warp's share of the items left.  Items cost from
// nothing (no image in the sweep) to 16,384 pairs, so a large claim of full items
// can outlast everything else (2: triclinic N = 200,000 9.9 ms; 3: 8.4; 6: 6.7;
// 12: 7.3), a small one pays for its run's setup (orthorhombic N = 100,000 2: 3.20,
// 6: 3.09, 12: 3.72, 24: 3.98 ms).
constexpr long long kClaims = 6;
constexpr unsigned kFlushPairs = 1u << 23;  // flush after this many i runs x images (2^30 pairs); a power of two

// A position: high parts on the frame's grid, sums of which are exact, and the rest.
struct Pos {
  float3 h, l;
};
__device__ __forceinline__ Pos unpack(float4 a, float2 b) {
  return Pos{make_float3(a.x, a.y, a.z), make_float3(a.w, b.x, b.y)};
}
// An i run: centre (on the grid), half extents, window W = c1 A + c0 (list_setup).
struct RunState {
  float3 c, h;
  float c1, c0;
};

// One warp's list: slot s holds y and W - |y|^2 of an image in pair layout (A: x,
// x', y, y'; B: z, z', and the last for slots 2p, 2p+1), the mask of each group
// of 8 slots and lane (bit 4 u + r: slot u of the group, i particle lane + 32 r),
// the queue of pairs to re-decide (reference, i particle), and the current i run.
// The ring holds a block waiting to fill plus one round of 32 appends.
template <int BLK>
struct WarpList {
  static constexpr int kCap = 2 * BLK;
  float4 A[kCap / 2];
  float4 B[kCap / 2];
  uint32_t ref[kCap];
  uint32_t mask[BLK / 8][32];
  uint2 queue[kQueueCap];
  RunState R;
  Pos o;  // the current image's origin
  unsigned long long uni, axis, cull;  // pairs, for the statistics
};
// Images of particles whose nearest image differs within the run (pick_round):
// y, W - |y|^2, and reference with kLastImage on a particle's last.
struct PickList {
  float4 M[kPickCap];
  uint32_t mref[kPickCap];
};
static_assert((sizeof(PickList) + sizeof(WarpList<kBlk>) - sizeof(WarpList<kBlkNarrow>)) * (kListBlock / 32) ==
                  4 * kPickWords, "shared memory of the shortest images, whose lists are the wide ones");

// What a block's pairs have in common (its segment), in shared memory.
struct SegState {
  FrameDev* F;
  const float4 *P4i, *P4j, *bi, *bj;  // positions and run bounds of the i and the j species
  const float2 *P2i, *P2j;
  int i0, j0, ni, nj, n_ti, n_tj, intra;
  int split, split_log2, part;  // items per run pair, j particles of an item
  int lo, hi;             // the sweep's bins
  float rc_hi2, rc_lo2;   // images kept: nearest distance^2 <= rc_hi2, farthest^2 >= rc_lo2
  float in_hi2, in_lo2;   // every pair in the sweep: farthest^2 <= in_hi2, nearest^2 >= in_lo2
  float grid, c0, abs, mid;  // FrameDev list_grid, list_c0, cull_abs, list_mid
  float nbins;
  int n_img, all, slow;   // images of a particle; FrameDev list_all; 1: list_slow, 2: some runs are far (slow_item)
  int inner;              // FrameDev in_range: nearly every block is an inner one
  long long items, item_base;
  long long claimers;     // claims that share the items left: kClaims per warp of the launch (or of the block)
  unsigned long long* next;
  uint64_t* out;          // the sweep's bins of the species pair's histogram
  float4 V4[27];  // image vectors: high parts on the grid and the rest of x,
  float2 V2[27];  //   the rest of y and z
};

// What a block keeps between its segments, in shared memory.
struct BlockState {
  int seg, len;                  // the segment, and the warps' first claims
  int next;                      // the segment to go on with, -1: none of its own left; known once asked
  unsigned since, asked;
  unsigned long long best, own;  // own: items claimed of a segment of its own
  long long base, first, seen;   // first claim, items known to be claimed
};

// d + l as a double-float (d a multiple of the grid, |l| about a step at most).
__device__ __forceinline__ DF renorm(float d, float l) {
  const float h = __fadd_rn(d, l);
  return {h, __fadd_rn(__fsub_rn(d, h), l)};
}

// |v|^2 - (c1 |v|^2 + c0) of a double-float vector, rounded once (to second order).
__device__ __forceinline__ float norm2_less(DF x, DF y, DF z, float c1, float c0) {
  const DF px = two_prod(x.h, x.h), py = two_prod(y.h, y.h), pz = two_prod(z.h, z.h);
  const DF s1 = two_sum(px.h, py.h);
  const DF s2 = two_sum(s1.h, pz.h);
  float low = __fmaf_rn(x.h + x.h, x.l, px.l);
  low = __fadd_rn(low, __fmaf_rn(y.h + y.h, y.l, py.l));
  low = __fadd_rn(low, __fmaf_rn(z.h + z.h, z.l, pz.l));
  low = __fadd_rn(low, __fadd_rn(s1.l, s2.l));
  return __fadd_rn(s2.h, __fsub_rn(low, __fmaf_rn(c1, s2.h, c0)));
}

// One run's state from its bounds (explicit roundings: the drain computes it
// again, and must get the same).  The window takes l of list_setup as
// H over three quarters of the sweep's end; 2^-7 covers the second-order terms and
// the rounding of W itself.
__device__ __forceinline__ RunState run_state(const SegState& G, float4 lo4, float4 hi4) {
  const float grid = G.grid;
  RunState r;
  r.c = make_float3(on_grid(__fmul_rn(0.5f, __fadd_rn(lo4.x, hi4.x)), grid),
                    on_grid(__fmul_rn(0.5f, __fadd_rn(lo4.y, hi4.y)), grid),
                    on_grid(__fmul_rn(0.5f, __fadd_rn(lo4.z, hi4.z)), grid));
  // (the bounds are those of the high parts)
  r.h = make_float3(__fadd_ru(fmaxf(__fsub_ru(hi4.x, r.c.x), __fsub_ru(r.c.x, lo4.x)), grid),
                    __fadd_ru(fmaxf(__fsub_ru(hi4.y, r.c.y), __fsub_ru(r.c.y, lo4.y)), grid),
                    __fadd_ru(fmaxf(__fsub_ru(hi4.z, r.c.z), __fsub_ru(r.c.z, lo4.z)), grid));
  const float H2 = __fmaf_ru(r.h.z, r.h.z, __fmaf_ru(r.h.y, r.h.y, __fmul_ru(r.h.x, r.h.x)));
  const float u = 0x1p-24f * (1.0f + 0x1p-7f);
  const float l = fminf(fmaxf(__fdiv_rn(__fsqrt_rn(H2), __fmul_rn(0.75f, (float)G.hi)), 0.01f), 2.0f);
  r.c1 = __fadd_rn(__fmul_rn(u, __fmaf_rn(6.0f, l, 2.0f)), 0x1p-27f);
  r.c0 = __fmaf_rn(__fmul_rn(u, __fadd_rn(5.0f, __fdiv_rn(6.0f, l))), H2, G.c0);
  return r;
}

// An i particle relative to the run's centre c: (2 x, -|x|^2), the factors of
// the FMA chain.
__device__ __forceinline__ float4 i_factors(const Pos& p, float3 c) {
  const DF x = renorm(__fsub_rn(p.h.x, c.x), p.l.x), y = renorm(__fsub_rn(p.h.y, c.y), p.l.y),
           z = renorm(__fsub_rn(p.h.z, c.z), p.l.z);
  return make_float4(2.0f * x.h, 2.0f * y.h, 2.0f * z.h, -norm2_less(x, y, z, 0.0f, 0.0f));
}

// The vector that takes a home position to image m relative to the centre c
// (itself on the grid).
__device__ __forceinline__ Pos image_vector(const FrameDev& F, int m, float grid) {
  Pos v;
  v.h = make_float3(on_grid(F.img_h[m][0], grid), on_grid(F.img_h[m][1], grid), on_grid(F.img_h[m][2], grid));
  v.l = make_float3(__fadd_rn(__fsub_rn(F.img_h[m][0], v.h.x), F.img_l[m][0]),
                    __fadd_rn(__fsub_rn(F.img_h[m][1], v.h.y), F.img_l[m][1]),
                    __fadd_rn(__fsub_rn(F.img_h[m][2], v.h.z), F.img_l[m][2]));
  return v;
}
__device__ __forceinline__ Pos image_origin(const SegState& G, int m, float3 c) {
  Pos o = unpack(G.V4[m], G.V2[m]);
  o.h = make_float3(__fsub_rn(o.h.x, c.x), __fsub_rn(o.h.y, c.y), __fsub_rn(o.h.z, c.z));
  return o;
}

// A listed image: (y, W - |y|^2).  With W added, q' = q - W takes the place of q:
// the sign of e' = n^2 - q' decides as that of n^2 - q does outside the window,
// and every pair inside it (0 <= e' <= 2 W) is counted one below the edge n.
__device__ __forceinline__ float4 j_image(const Pos& p, const Pos& o, float c1, float c0) {
  const DF x = renorm(__fadd_rn(p.h.x, o.h.x), __fadd_rn(p.l.x, o.l.x)),
           y = renorm(__fadd_rn(p.h.y, o.h.y), __fadd_rn(p.l.y, o.l.y)),
           z = renorm(__fadd_rn(p.h.z, o.h.z), __fadd_rn(p.l.z, o.l.z));
  return make_float4(x.h, y.h, z.h, -norm2_less(x, y, z, c1, c0));
}

// ------------------------------------------------------------------ re-decision

// The definition's bin of one pair, counted only when its nearest image is the
// listed one (displacement d): nbins when it is another.  For the frames whose
// images are not listed (any), whatever the image.
template <int V>
__device__ __forceinline__ int exact_listed(const FrameDev& F, int i, int j, float3 d, bool any) {
  const double3 pi = coords64(F, i), pj = coords64(F, j);
  if (V != V_NONE && !any) {
    const double3 e = exact_image<V>(F, pi, pj);
    if (!(fabsf((float)e.x * F.S - d.x) < 0.5f * F.period[0] && fabsf((float)e.y * F.S - d.y) < 0.5f * F.period[1] &&
          fabsf((float)e.z * F.S - d.z) < 0.5f * F.period[2]))
      return F.nbins;
  }
  return bin_from_thresholds(F.T, F.S, F.nbins, exact_r2<V>(F, pi, pj));
}
__device__ __noinline__ int exact_listed_bin(const FrameDev& F, int i, int j, float3 d, bool any) {
  return F.variant == V_NONE    ? exact_listed<V_NONE>(F, i, j, d, any)
         : F.variant == V_ORTHO ? exact_listed<V_ORTHO>(F, i, j, d, any)
         : F.variant == V_TRIC ? exact_listed<V_TRIC>(F, i, j, d, any)
                               : exact_listed<V_TRIC_SEARCH>(F, i, j, d, true);
}

// Bin of a re-decided pair (particles i and j of the segment's species) from q in double-float arithmetic (about 44 bits) for
// the listed image m, and the integer n nearest to its root.  An image inside r_max
// is the definition's: the shortest by a margin (F.pick), else the only one there
// (check_frame), up to ties of two at r_max itself.  When q is too close to n^2, or the
// image is not known (m < 0), the binary64 replay decides.
__device__ __forceinline__ int listed_bin(const SegState& G, int i, int j, int m, float& n, unsigned& nexact) {
  const Pos a = unpack(__ldg(G.P4i + i), __ldg(G.P2i + i)), b = unpack(__ldg(G.P4j + j), __ldg(G.P2j + j));
  const float ah[3] = {a.h.x, a.h.y, a.h.z}, al[3] = {a.l.x, a.l.y, a.l.z};
  const float bh[3] = {b.h.x, b.h.y, b.h.z}, bl[3] = {b.l.x, b.l.y, b.l.z};
  const Pos v = unpack(G.V4[max(m, 0)], G.V2[max(m, 0)]);
  const float vh[3] = {v.h.x, v.h.y, v.h.z}, vl[3] = {v.l.x, v.l.y, v.l.z};
  DF d[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    d[c] = two_sum(__fadd_rn(__fsub_rn(bh[c], ah[c]), vh[c]), __fadd_rn(vl[c], __fsub_rn(bl[c], al[c])));
  }
  const DF q = df_norm2(d[0], d[1], d[2]);
  const float s = sqrt_approx(q.h);
  n = nint_f(s);
  const DF n2 = two_prod(n, n);
  const float diff = __fadd_rn(__fsub_rn(q.h, n2.h), __fsub_rn(q.l, n2.l));
  // 2^-38: the double-float arithmetic and the binary64 rounding of the definition;
  // at r_max also the images that tie at half a period, 2^-40 of it within r_max (check_frame)
  const float rel = n >= G.nbins ? 0x1p-36f : 0x1p-38f;
  if (m >= 0 && (fabsf(diff) > __fmaf_rn(rel, q.h, G.mid * s) + 0x1p-60f || n < 0.5f))
    return (int)fminf(n, G.nbins + 1.0f) - (diff < 0.0f && n >= 0.5f ? 1 : 0);
  ++nexact;
  return exact_listed_bin(*G.F, G.i0 + i, G.j0 + j, make_float3(d[0].h, d[1].h, d[2].h), G.F->pick != 0);
}

// The shortest image of a pair in float32, -1 if another comes within 2^-16 of it.
__device__ __noinline__ int picked_image(const FrameDev& F, int i, int j) {
  const Pos a = unpack(__ldg(F.P4 + i), __ldg(F.P2 + i)), b = unpack(__ldg(F.P4 + j), __ldg(F.P2 + j));
  const float dx = b.h.x - a.h.x, dy = b.h.y - a.h.y, dz = b.h.z - a.h.z;
  float best = INFINITY, next = INFINITY;
  int m = kHome;
  for (int k = 0; k < 27; ++k) {
    const float x = dx + F.img_h[k][0], y = dy + F.img_h[k][1], z = dz + F.img_h[k][2];
    const float q = x * x + y * y + z * z;
    next = fminf(next, fmaxf(q, best));
    if (q < best) {
      best = q;
      m = k;
    }
  }
  // (the low parts and the roundings move a distance by less than cull_abs)
  const float slack = 4.0f * F.cull_abs * (sqrtf(next) + F.cull_abs);
  return next - best > best * 0x1p-16f + slack ? m : -1;
}

__device__ float4 run_factor(const SegState& G, int i, int end, float3 c);

// The word in which the pair loop counted a pair close to its run (q' below
// (2 W + 1)^2 or nearly): the scalar replay of its float32 arithmetic.
__device__ __noinline__ int replay_rel(const SegState& G, int i, int j, int m) {
  const FrameDev& F = *G.F;
  const RunState R = run_state(G, __ldg(G.bi + 2 * (i / kRun)), __ldg(G.bi + 2 * (i / kRun) + 1));
  const float4 x = run_factor(G, i, i + 1, R.c);
  const float4 y = j_image(unpack(__ldg(G.P4j + j), __ldg(G.P2j + j)), image_origin(G, m, R.c), R.c1, R.c0);
  const float nq = __fadd_rn(__fmaf_rn(y.x, x.x, __fmaf_rn(y.y, x.y, __fmaf_rn(y.z, x.z, x.w))), y.w);
  const int lane = i & 31;
  float sc = fminf(sqrt_approx(-nq), (float)(G.hi + 1 + lane));
  if (G.lo > 0) sc = fmaxf(sc, (float)(G.lo - lane));
  const float sm = __fadd_rn(sc, kMagicRound);
  const float n = __fadd_rn(sm, -kMagicRound);
  const float e = __fmaf_rn(n, n, nq);
  return __float_as_int(sm) + (int)(__float_as_uint(e) >> 31) - (__float_as_int(kMagicRound) + G.lo + 1);
}

// Re-decisions are few and dear: 0.1 to 3 % of the pairs, each the time of about 25
// pairs of the loop, most of it the latency of the four gathers and of fetching code
// that is seldom run.  So it is one piece of straight code (with two calls, an image
// vector formed from the descriptor per pair, and a binary64 replay for every image
// at half a period: 50 to 95 pairs; N = 30,000 triclinic, 73,770 bins 1.99 -> 0.95 ms),
// and pairs are re-decided for their own image's window only (below (2 W + 1)^2 at the
// far corner of the run's box: 0.95 ms, of their own image 0.62).
// Decide the first min(32, qcount) queued pairs (reference, i particle), one per
// lane, and shift the rest of the queue down.  A pair was counted one below its
// edge n and moves up when it belongs there; close to the run, where the window
// may hold several edges, the word it was counted in is found by replay.
// Pairs with kAnyImage were not counted.
constexpr uint32_t kNearPair = 0x80000000u;
__device__ __noinline__ int list_drain(const SegState& G, uint2* q, int qcount, uint32_t* sh, int lane) {
  const int count = qcount < 32 ? qcount : 32;
  unsigned nexact = 0;
  __syncwarp();
  if (lane < count) {
    const uint2 e = q[lane];
    const int width = G.hi - G.lo;
    int m = (int)(e.x >> kImgShift);
    const int i = (int)(e.y & ~kNearPair), j = (int)(e.x & ((1u << kImgShift) - 1u));
    float n;
    int bin, prov;
    const bool any = e.x >= kAnyImage;
    if (any) m = picked_image(*G.F, G.i0 + i, G.j0 + j);
    bin = listed_bin(G, i, j, m, n, nexact) - G.lo;
    prov = any ? -1 : (int)n - 1 - G.lo;
    if (e.y & kNearPair) prov = replay_rel(G, i, j, m);
    if (bin != prov) {
      if ((uint32_t)bin < (uint32_t)width) atomicAdd(sh + bin, 1u);
      if ((uint32_t)prov < (uint32_t)width) atomicAdd(sh + prov, 0xFFFFFFFFu);
    }
  }
  __syncwarp();
  const int rest = qcount - count;
  const uint2 keep = lane < rest ? q[32 + lane] : make_uint2(0u, 0u);
  __syncwarp();
  if (lane < rest) q[lane] = keep;
  __syncwarp();
  for (int o = 16; o > 0; o >>= 1) nexact += __shfl_xor_sync(kFull, nexact, o);
  if (lane == 0) {
    atomicAdd(&G.F->deferred, (unsigned long long)count);
    if (nexact) atomicAdd(&G.F->exact, (unsigned long long)nexact);
  }
  return rest;
}

// ------------------------------------------------------------------ the pair loop

// This lane's four i particles, broadcast to both halves of a float32x2.
struct IRegs {
  float2 x[4], y[4], z[4], w[4];
};
// The factors of i particle i of the run with centre c, NaN beyond its end.  One
// copy of the arithmetic: the executed code has to stay in the instruction cache.
__device__ __noinline__ float4 run_factor(const SegState& G, int i, int end, float3 c) {
  const int k = min(i, end - 1);
  const float4 x = i_factors(unpack(__ldg(G.P4i + k), __ldg(G.P2i + k)), c);
  return i < end ? x : make_float4(NAN, NAN, NAN, NAN);
}
__device__ __forceinline__ void load_run(const SegState& G, float3 c, int i_begin, int ni, int lane, IRegs& I) {
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const float4 x = run_factor(G, i_begin + lane + 32 * r, i_begin + ni, c);
    I.x[r] = bc2(x.x);
    I.y[r] = bc2(x.y);
    I.z[r] = bc2(x.z);
    I.w[r] = bc2(x.w);
  }
}

// Count one pair: the word of bin n - 1 + signbit(e') of the sweep at byte
// address 4 v + hbase (v = bits(sm) + signbit), and the mask bit of a pair inside
// the window: 0 <= e' < w2 as unsigned bits (negative e' compare above, and NaN,
// e' or both, is not below).  NEAR: and of a pair with -nq < -nqm.
template <bool NEAR>
__device__ __forceinline__ void count_listed(float sm, float e, float nq, uint32_t w2, float nqm, uint32_t hbase,
                                             uint32_t bit, uint32_t& dmask) {
  if (NEAR)
    asm volatile(
        "{\n\t.reg .pred p, n;\n\t.reg .u32 sg, v, addr;\n\t"
        "shr.u32 sg, %2, 31;\n\t"
        "add.u32 v, %1, sg;\n\t"
        "mad.lo.u32 addr, v, 4, %4;\n\t"
        "setp.gt.f32 n, %6, %7;\n\t"
        "setp.lt.or.u32 p, %2, %3, n;\n\t"
        "@p or.b32 %0, %0, %5;\n\t"
        "red.shared.add.u32 [addr], 1;\n\t"
        "}"
        : "+r"(dmask)
        : "r"(__float_as_uint(sm)), "r"(__float_as_uint(e)), "r"(w2), "r"(hbase), "r"(bit), "f"(nq), "f"(nqm));
  else
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .u32 sg, v, addr;\n\t"
        "shr.u32 sg, %2, 31;\n\t"
        "add.u32 v, %1, sg;\n\t"
        "mad.lo.u32 addr, v, 4, %4;\n\t"
        "setp.lt.u32 p, %2, %3;\n\t"
        "@p or.b32 %0, %0, %5;\n\t"
        "red.shared.add.u32 [addr], 1;\n\t"
        "}"
        : "+r"(dmask)
        : "r"(__float_as_uint(sm)), "r"(__float_as_uint(e)), "r"(w2), "r"(hbase), "r"(bit));
}

// Queue the pairs whose mask bits are set (groups: this lane's groups with any;
// first: the run's first particle and flag):
// one per lane per turn, each lane from its own first group, so that a block
// takes two or three turns.
template <int BLK>
__device__ __forceinline__ int push_pairs(const SegState& G, WarpList<BLK>& W, int s0, uint32_t groups, uint32_t first,
                                          uint32_t* sh, int lane, int qcount) {
  unsigned bal = __ballot_sync(kFull, groups != 0u);
  while (bal) {
    if (groups) {
      const int g = __ffs(groups) - 1;
      const uint32_t m = W.mask[g][lane];
      const int b = __ffs(m) - 1;
      W.mask[g][lane] = m & (m - 1u);
      if ((m & (m - 1u)) == 0u) groups &= groups - 1u;
      W.queue[qcount + __popc(bal & ((1u << lane) - 1u))] =
          make_uint2(W.ref[s0 + 8 * g + (b >> 2)], first + (uint32_t)(lane + 32 * (b & 3)));
    }
    qcount += __popc(bal);
    if (qcount >= 32) qcount = list_drain(G, W.queue, qcount, sh, lane);
    bal = __ballot_sync(kFull, groups != 0u);
  }
  return qcount;
}

// Listed images [s0, s0 + n) (multiples of 8, within the ring) against the run of
// i particles from i_begin.  The root is clamped to the sweep, so that pairs
// outside it land in guard words, spread over the lanes, and outside the window;
// NaN (padding) becomes the upper clamp.  INNER: a whole block (no padding) of
// images all of whose pairs lie in the sweep, no clamp needed.  NEAR: images so near
// the run that q' may be below (2 W + 1)^2, where the window can hold several edges:
// those pairs are re-decided too (list_all: every pair); and with above >= 0, only
// particles j > above + i (the diagonal item of one species; else above = -2^30).
// Returns this lane's groups with pairs to re-decide.
enum BlockMode { PLAIN, INNER, NEARBY };
template <BlockMode MODE, bool MULTI, int BLK>
__device__ __forceinline__ uint32_t list_block(const SegState& G, const IRegs& I, WarpList<BLK>& W, int s0, int n, int above,
                                               uint32_t* sh, int lane) {
  constexpr bool NEAR = MODE == NEARBY;
  const int lo = G.lo, hi = G.hi;
  const uint32_t hbase =
      (uint32_t)__cvta_generic_to_shared(sh) - 4u * (uint32_t)(__float_as_int(kMagicRound) + lo + 1);
  const float chi = (float)(hi + 1 + lane), clo = (float)(lo - lane);
  const float2 M = bc2(kMagicRound), NM = bc2(-kMagicRound);
  // 2 W from W - A, rounded up: 2 (c1 A + c0) <= w1 (A - W) + w0
  const float2 w1 = bc2(-2.0f * W.R.c1 * (1.0f + 0x1p-10f)), w0 = bc2(2.0f * W.R.c0 * (1.0f + 0x1p-10f));
  uint32_t groups = 0u;
#pragma unroll 1
  for (int g = 0; g < n; g += 8) {
    const int sg = s0 + g;
    uint32_t dmask = 0u;
#pragma unroll(NEAR ? 1 : 4)
    for (int u = 0; u < 8; u += 2) {
      const float4 A = W.A[(sg + u) >> 1], Bv = W.B[(sg + u) >> 1];
      const float2 yx = make_float2(A.x, A.y), yy = make_float2(A.z, A.w), yz = make_float2(Bv.x, Bv.y),
                   na = make_float2(Bv.z, Bv.w);
      const float2 w2 = fma2(na, w1, w0);
      int ja = 0, jb = 0;
      float2 qm = bc2(0.0f);
      if (NEAR) {
        const float2 r = add2(w2, bc2(1.0f));
        qm = G.all ? bc2(INFINITY) : mul2(r, r);
        ja = (int)(W.ref[sg + u] & ((1u << kImgShift) - 1u)) - above - lane;
        jb = (int)(W.ref[sg + u + 1] & ((1u << kImgShift) - 1u)) - above - lane;
      }
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        float2 nq = add2(fma2(yx, I.x[r], fma2(yy, I.y[r], fma2(yz, I.z[r], I.w[r]))), na);
        if (NEAR) {
          if (ja <= 32 * r) nq.x = NAN;
          if (jb <= 32 * r) nq.y = NAN;
        }
        float2 sc = make_float2(sqrt_approx(-nq.x), sqrt_approx(-nq.y));
        if (MODE != INNER) {
          sc = make_float2(fminf(sc.x, chi), fminf(sc.y, chi));
          if (MULTI) sc = make_float2(fmaxf(sc.x, clo), fmaxf(sc.y, clo));
        }
        const float2 sm = add2(sc, M);
        const float2 nn = add2(sm, NM);
        const float2 e = fma2(nn, nn, nq);
        count_listed<NEAR>(sm.x, e.x, nq.x, __float_as_uint(w2.x), -qm.x, hbase, 1u << (u * 4 + r), dmask);
        count_listed<NEAR>(sm.y, e.y, nq.y, __float_as_uint(w2.y), -qm.y, hbase, 1u << ((u + 1) * 4 + r), dmask);
      }
    }
    W.mask[g >> 3][lane] = dmask;
    if (dmask) groups |= 1u << (g >> 3);
  }
  return groups;
}

// The near form out of line (it loads the run again) and not unrolled.
template <bool MULTI, int BLK>
__device__ __noinline__ uint32_t list_near(const SegState& G, WarpList<BLK>& W, int i_begin, int ni, int s0, int n,
                                           int above, uint32_t* sh, int lane) {
  IRegs I;
  load_run(G, W.R.c, i_begin, ni, lane, I);
  return list_block<NEARBY, MULTI>(G, I, W, s0, n, above, sh, lane);
}

// Frames whose r_max exceeds half the distance between images (F.pick): a pair's
// distance is the shortest over the images, so an image of a particle is listed
// alone only when it is the shortest for every particle of the run.
//
// One round of 32 j particles (this lane's at p, index jl, if valid) of a j run of
// which several images (mask) can be the shortest for some pair.  Per particle,
// an image whose nearest distance to the run's box exceeds another's farthest
// cannot be.  Returns the image of a particle left with one, else -1.  The others'
// images are evaluated here, the smallest q' = q - W taken over them: with W the
// largest of theirs, the pair's q lies in [q', q' + 2 W], as for a single image.
// Pairs inside the window or below (2 W + 1)^2 go to a guard word and to the queue,
// to be counted by the drain.
template <bool MULTI>
__device__ __noinline__ int pick_round(const SegState& G, WarpList<kBlk>& W, PickList& K, unsigned mask, Pos p, int jl, bool valid,
                                       int i_begin, int ni, int above, uint32_t* sh, int lane, int& qcount) {
  const FrameDev& F = *G.F;
  const float3 h = W.R.h;
  float far = INFINITY;
  bool below = false;  // some image has every pair below the sweep: so has the shortest
  for (unsigned k = mask; k; k &= k - 1u) {
    const Pos o = image_origin(G, __ffs(k) - 1, W.R.c);
    const float x = fabsf(p.h.x + o.h.x) + h.x, y = fabsf(p.h.y + o.h.y) + h.y, z = fabsf(p.h.z + o.h.z) + h.z;
    const float f = x * x + y * y + z * z;
    far = fminf(far, f);
    if (MULTI) below = below || f < G.rc_lo2;
  }
  const float reach = sqrtf(far) * (1.0f + 0x1p-15f) + G.abs;
  const float lim = fminf(reach * reach, G.rc_hi2);
  unsigned cand = 0u;
  if (valid && !below)
    for (unsigned k = mask; k; k &= k - 1u) {
      const Pos o = image_origin(G, __ffs(k) - 1, W.R.c);
      const float x = fmaxf(fabsf(p.h.x + o.h.x) - h.x, 0.0f), y = fmaxf(fabsf(p.h.y + o.h.y) - h.y, 0.0f),
                  z = fmaxf(fabsf(p.h.z + o.h.z) - h.z, 0.0f);
      if (x * x + y * y + z * z <= lim) cand |= k & (0u - k);
    }
  const int single = __popc(cand) == 1 ? __ffs(cand) - 1 : -1;
  if (single >= 0) cand = 0u;
  if (!__any_sync(kFull, cand != 0u)) return single;

  IRegs I;
  load_run(G, W.R.c, i_begin, ni, lane, I);
  float2 x2[2], y2[2], z2[2], w2[2];  // factors of i particles (0, 1) and (2, 3)
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    x2[r] = make_float2(I.x[2 * r].x, I.x[2 * r + 1].x);
    y2[r] = make_float2(I.y[2 * r].x, I.y[2 * r + 1].x);
    z2[r] = make_float2(I.z[2 * r].x, I.z[2 * r + 1].x);
    w2[r] = make_float2(I.w[2 * r].x, I.w[2 * r + 1].x);
  }
  const float chi = (float)(G.hi + 1 + lane), clo = (float)(G.lo - lane);
  const float v1 = -2.0f * W.R.c1 * (1.0f + 0x1p-10f), v0 = 2.0f * W.R.c0 * (1.0f + 0x1p-10f);
  const int first = __float_as_int(kMagicRound) + G.lo + 1;
  while (__any_sync(kFull, cand != 0u)) {
    // as many of the particles left, in lane order, as fit
    const int c = __popc(cand);
    int end = c;
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(kFull, end, o);
      if (lane >= o) end += t;
    }
    const bool now = c > 0 && end <= kPickCap;
    const int count = __reduce_max_sync(kFull, end <= kPickCap ? end : 0);
    if (now) {
      int s = end - c;
      for (; cand; cand &= cand - 1u, ++s) {
        const int m = __ffs(cand) - 1;
        K.M[s] = j_image(p, image_origin(G, m, W.R.c), W.R.c1, W.R.c0);
        K.mref[s] = (uint32_t)jl | (s == end - 1 ? kLastImage : 0u);
      }
    }
    __syncwarp();
    float2 nq[2] = {bc2(-INFINITY), bc2(-INFINITY)};
    float win = 0.0f;
    for (int s = 0; s < count; ++s) {
      const float4 y = K.M[s];
      const uint32_t ref = K.mref[s];
      win = fmaxf(win, __fmaf_rn(y.w, v1, v0));
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        const float2 t =
            add2(fma2(bc2(y.x), x2[r], fma2(bc2(y.y), y2[r], fma2(bc2(y.z), z2[r], w2[r]))), bc2(y.w));
        nq[r] = make_float2(fmaxf(nq[r].x, t.x), fmaxf(nq[r].y, t.y));
      }
      if (!(ref & kLastImage)) continue;
      const int j = (int)(ref & ~kLastImage);
      const float qm = G.all ? INFINITY : __fmul_rn(win + 1.0f, win + 1.0f);
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const float v = (r & 1) ? nq[r >> 1].y : nq[r >> 1].x;
        const int il = lane + 32 * r;
        const bool ok = il < ni && j > above + il;
        float sc = fminf(sqrt_approx(fabsf(v)), chi);
        if (MULTI) sc = fmaxf(sc, clo);
        const float sm = __fadd_rn(sc, kMagicRound);
        const float n = __fadd_rn(sm, -kMagicRound);
        const float e = __fmaf_rn(n, n, v);
        const bool defer = ok && (-v < qm || __float_as_uint(e) < __float_as_uint(win));
        const int rel = __float_as_int(sm) + (int)(__float_as_uint(e) >> 31) - first;
        atomicAdd(sh + (ok && !defer ? rel : G.hi - G.lo + lane), 1u);
        const unsigned bal = __ballot_sync(kFull, defer);
        if (bal) {
          if (defer)
            W.queue[qcount + __popc(bal & ((1u << lane) - 1u))] =
                make_uint2((uint32_t)j | kAnyImage, (uint32_t)(i_begin + il));
          qcount += __popc(bal);
          if (qcount >= 32) qcount = list_drain(G, W.queue, qcount, sh, lane);
        }
      }
      nq[0] = nq[1] = bc2(-INFINITY);
      win = 0.0f;
    }
    __syncwarp();
  }
  return single;
}

// Of two runs of which one is far (FrameDev.list_far): the gap between their bounds puts
// every pair beyond the sweep (2^-20 of the coordinates for the rounding of the bounds).
__device__ __forceinline__ bool far_apart(const SegState& G, float4 ilo, float4 ihi, float4 jlo, float4 jhi) {
  auto gap = [](float il, float ih, float jl, float jh) {
    const float size = fmaxf(fmaxf(fabsf(il), fabsf(ih)), fmaxf(fabsf(jl), fabsf(jh)));
    return fmaxf(fmaxf(jl - ih, il - jh) - size * 0x1p-20f, 0.0f);
  };
  const float gx = gap(ilo.x, ihi.x, jlo.x, jhi.x), gy = gap(ilo.y, ihi.y, jlo.y, jhi.y),
              gz = gap(ilo.z, ihi.z, jlo.z, jhi.z);
  return gx * gx + gy * gy + gz * gz > G.rc_hi2;
}

// Bin of a pair without a box from its float32 coordinates, -1 when their rounding leaves
// it open.  The differences in bins err by 3 u (u = 2^-24) of themselves wherever the
// particles are, their squares' sum by less than 10 u: 2^-19 is far on the safe side.
__device__ __noinline__ int far_pair_bin(const FrameDev& F, int i, int j) {
  const float4 a = __ldg(F.X + i), b = __ldg(F.X + j);
  const float x = __fmul_rn(__fsub_rn(b.x, a.x), F.S), y = __fmul_rn(__fsub_rn(b.y, a.y), F.S),
              z = __fmul_rn(__fsub_rn(b.z, a.z), F.S);
  const float q = __fmaf_rn(z, z, __fmaf_rn(y, y, __fmul_rn(x, x)));
  const float s = sqrt_approx(q);
  if (s > (float)F.nbins + 1.0f + (float)F.nbins * 0x1p-18f) return F.nbins;  // (infinities too)
  const float n = nint_f(s), e = __fmaf_rn(n, n, -q);
  if (n >= 0.5f && fabsf(e) <= q * 0x1p-19f) return -1;
  return (int)n - (e > 0.0f ? 1 : 0);
}

// Every pair of an item in binary64, in frames whose images cannot be listed (G.slow 1)
// or for a far run (G.slow 2, i run ri and j run rj; float32 where it is enough: one far
// particle of N = 100,000 takes a run's 1.3e7 pairs here, 1.2 ms of binary64).  Returns the images that the item
// counts for towards the flush, -1 for an item of two runs that are not far: nothing done.
__device__ __noinline__ int slow_item(const SegState& G, int ri, int rj, int ni, int jbeg, int jend, uint32_t* sh, int lane) {
  if (G.slow == 2) {
    const float4 ilo = __ldg(G.bi + 2 * ri), ihi = __ldg(G.bi + 2 * ri + 1);
    const float4 jlo = __ldg(G.bj + 2 * rj), jhi = __ldg(G.bj + 2 * rj + 1);
    if (ilo.w == 0.0f && jlo.w == 0.0f) return -1;
    if (far_apart(G, ilo, ihi, jlo, jhi)) return 0;
  }
  FrameDev* const Fp = G.F;
  const int ib = ri * kRun, nj = jend - jbeg;
  // (up to 2^18 bins the root's error leaves the nearest integer right to within one)
  const bool fast = G.slow == 2 && !Fp->X64 && Fp->nbins <= (1 << 18);
  unsigned long long np = 0;
  for (int p = lane; p < ni * nj; p += 32) {
    const int i = ib + p % ni, j = jbeg + p / ni;
    if (G.intra && j <= i) continue;
    int bin = fast ? far_pair_bin(*Fp, G.i0 + i, G.j0 + j) : -1;
    if (bin < 0) {
      bin = exact_listed_bin(*Fp, G.i0 + i, G.j0 + j, make_float3(0.f, 0.f, 0.f), true);
      ++np;
    }
    const int rel = bin - G.lo;
    if ((uint32_t)rel < (uint32_t)(G.hi - G.lo)) atomicAdd(sh + rel, 1u);
  }
  for (int o = 16; o > 0; o >>= 1) np += __shfl_xor_sync(kFull, np, o);
  if (lane == 0 && np) {
    atomicAdd(&Fp->deferred, np);
    atomicAdd(&Fp->exact, np);
  }
  return kRun;
}

// Adds one word's count to the global histogram.  Counts are signed: a
// provisional count may be moved after the words were flushed.
__device__ __forceinline__ void merge_count(uint64_t* dst, uint32_t v) {
  if (v) atomicAdd((unsigned long long*)dst, (unsigned long long)(long long)(int32_t)v);
}

// One thread fills the block's segment state, but for the item counter.
__device__ void enter_segment(const ListSegment& S, SegState& G) {
  FrameDev* const Fp = S.fd;
  const FrameDev& F = *Fp;
  G.F = Fp;
  G.P4i = F.P4 + S.i0;
  G.P4j = F.P4 + S.j0;
  G.P2i = F.P2 + S.i0;
  G.P2j = F.P2 + S.j0;
  G.bi = F.bnd + 2 * S.i_run0;
  G.bj = F.bnd + 2 * S.j_run0;
  G.i0 = S.i0;
  G.j0 = S.j0;
  G.ni = S.ni;
  G.nj = S.nj;
  G.n_ti = S.n_ti;
  G.n_tj = S.n_tj;
  G.intra = S.intra;
  G.split_log2 = S.split_log2;
  G.split = 1 << S.split_log2;
  G.part = kRun >> S.split_log2;
  G.lo = S.pass * F.sweep_width;
  G.hi = min(F.nbins, G.lo + F.sweep_width);
  // widened (or narrowed) by 2^-15 and the absolute slack for the float32
  // roundings of the bounds and the binary64 rounding of the bin
  const float up = 1.0f + 0x1p-15f, down = 1.0f - 0x1p-15f;
  const float r_hi = (float)G.hi * up + F.cull_abs, r_lo = fmaxf((float)G.lo * down - F.cull_abs, 0.0f);
  const float n_hi = fmaxf((float)G.hi * down - F.cull_abs, 0.0f), n_lo = G.lo > 0 ? (float)G.lo * up + F.cull_abs : 0.0f;
  G.rc_hi2 = r_hi * r_hi;
  G.rc_lo2 = r_lo * r_lo;
  G.in_hi2 = n_hi * n_hi;
  G.in_lo2 = n_lo * n_lo;
  G.grid = F.list_grid;
  G.c0 = F.list_c0;
  G.abs = F.cull_abs;
  G.mid = F.list_mid;
  G.nbins = (float)F.nbins;
  G.n_img = F.variant == V_NONE ? 1 : 27;
  G.all = F.list_all;
  G.slow = F.list_slow ? 1 : F.list_far < INFINITY ? 2 : 0;
  // elsewhere the two loops would take turns in the instruction cache, at a loss
  G.inner = F.in_range;
  G.items = (G.lo < F.nbins && !F.bad) ? S.items : 0;
  G.item_base = S.item_base;
  G.out = F.out + (size_t)S.h * F.nbins + G.lo;
}

// The work distribution keeps its state in shared memory: whatever of it is in a register
// across the pair loop is spilled there (as local variables 196 bytes of spills instead
// of 132, and 1 % of every frame's time).

// The next segment that is one block's own, -1 when all are handed out.
__device__ __forceinline__ int own_segment(const ListLaunch& L) {
  if (L.n_shared == L.n_segs) return -1;
  const unsigned long long t = atomicAdd(&L.ctr[L.n_shared].next, 1ull);
  return t < (unsigned long long)(L.n_segs - L.n_shared) ? L.n_shared + (int)t : -1;
}

// Some blocks start spread over the shared segments' items, the others with segments of
// their own (one thread).
__device__ __forceinline__ int first_segment(const ListLaunch& L) {
  int own = -1;
  if ((int)blockIdx.x >= L.shared_blocks) own = own_segment(L);
  if (own >= 0 || L.n_shared == 0) return own;
  const double part = (double)blockIdx.x / ((int)blockIdx.x < L.shared_blocks ? L.shared_blocks : (int)gridDim.x);
  const long long pos = (long long)((double)L.shared_items * part);
  int lo = 0, hi = L.n_shared - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (L.segs[mid].item0 <= pos) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// One thread attaches the block to segment B.seg and makes the first claim for all its
// warps; claims shrink with the items left (a kClaims'th of an even share of them), at
// first at most the block's share of the launch.
__device__ __forceinline__ void attach_segment(const ListLaunch& L, BlockState& B, SegState& G) {
  constexpr int kWarps = kListBlock / 32;
  const int seg = B.seg;
  const bool shared = seg < L.n_shared;
  if (shared) atomicAdd(&L.ctr[seg].attached, 1);
  enter_segment(L.segs[seg], G);
  G.next = shared ? &L.ctr[seg].next : &B.own;
  G.claimers = kClaims * kWarps * (shared ? (long long)gridDim.x : 1LL);
  B.own = 0ull;
  B.asked = 0u;
  B.next = -1;
  const long long part = max(1LL, min(G.items / G.claimers, 1024LL));
  const long long share = max(1LL, (L.n_items + gridDim.x - 1) / (long long)gridDim.x);
  const long long want = min(part * kWarps, share);
  B.len = (int)part;
  B.first = want;
  B.base = G.items ? (long long)atomicAdd(G.next, (unsigned long long)want) : 0LL;
  B.seen = B.base + want;
  B.since = 0u;
}

// The block leaves its segment for B.next, or for the shared segment with the most work
// left per block; of several, each block takes the first after its own place.
__device__ __forceinline__ void next_segment(const ListLaunch& L, BlockState& B, const SegState& G, int tid, int lane) {
  const int next = B.next;
  if (tid == 0) {
    const int seg = B.seg;
    B.best = 0ull;
    B.seg = next;
    if (seg < L.n_shared) {
      atomicAdd(&L.ctr[seg].attached, -1);
      if (!G.items) L.ctr[seg].next = (unsigned long long)L.segs[seg].items;  // nothing to do for anyone
    }
  }
  __syncthreads();
  if (next >= 0) return;
  const int place = (int)((long long)L.n_shared * blockIdx.x / gridDim.x);
  unsigned long long best = 0ull;
  for (int k = tid; k < L.n_shared; k += kListBlock) {
    const int at = k + place < L.n_shared ? k + place : k + place - L.n_shared;
    const unsigned long long nx = *(volatile unsigned long long*)&L.ctr[at].next;
    const unsigned long long it = (unsigned long long)L.segs[at].items;
    if (nx >= it) continue;
    const int att = *(volatile int32_t*)&L.ctr[at].attached;
    unsigned long long score = (it - nx) * 16ull / (unsigned long long)(1 + max(att, 0));
    score = min(max(score, 1ull), (1ull << 40) - 1ull);
    best = max(best, (score << 24) | (unsigned long long)(L.n_shared - 1 - k));
  }
  for (int o = 16; o > 0; o >>= 1) best = max(best, __shfl_xor_sync(kFull, best, o));
  if (lane == 0 && best) atomicMax(&B.best, best);
  __syncthreads();
  if (tid == 0 && B.best) {
    const int at = L.n_shared - 1 - (int)(B.best & 0xFFFFFFull) + place;
    B.seg = at < L.n_shared ? at : at - L.n_shared;
  }
  __syncthreads();
}

// Item -> (i run, j run, part).  Row a of a species with itself starts at item
// a n - a (a - 1) / 2; the row is found from the root of that (the discriminant
// is exact, its float32 root within a row of the truth).
__device__ __forceinline__ void item_of(const SegState& G, long long u, int& ri, int& rj, int& sub) {
  const long long v = u + G.item_base, lid = v >> G.split_log2;
  sub = (int)v & (G.split - 1);
  if (G.intra) {
    const long long n = G.n_tj, t = 2 * n + 1;
    int a = (int)(0.5f * ((float)t - sqrtf((float)max(t * t - 8 * lid, 0LL))));
    a = min(max(a, 0), G.n_ti - 1);
    while (a > 0 && a * n - (long long)a * (a - 1) / 2 > lid) --a;
    while (a + 1 < G.n_ti && (a + 1) * n - (long long)(a + 1) * a / 2 <= lid) ++a;
    ri = a;
    rj = a + (int)(lid - (a * n - (long long)a * (a - 1) / 2));
  } else {
    ri = (int)(lid / G.n_tj);
    rj = (int)(lid - (long long)ri * G.n_tj);
  }
}

// One block of 16 warps with 128 registers per SM: the pair loop and the list
// state stay in registers, and the SM merges one histogram per segment.
// PICK: frames whose pairs take the shortest of several images (pick_round).
// BLK: see kBlk (PICK: 64).
template <bool MULTI, bool PICK, int BLK>
__global__ void __launch_bounds__(kListBlock, 1) list_kernel(const __grid_constant__ ListLaunch L) {
  extern __shared__ __align__(16) unsigned char smem[];
  constexpr int BLOCK = kListBlock, kWarps = BLOCK / 32, kCap = 2 * BLK;
  WarpList<BLK>* lists = reinterpret_cast<WarpList<BLK>*>(smem);
  PickList* picks = reinterpret_cast<PickList*>(smem + sizeof(WarpList<BLK>) * kWarps);
  uint32_t* sh = reinterpret_cast<uint32_t*>(picks + (PICK ? kWarps : 0)) + kGuard;
  __shared__ BlockState B;
  __shared__ SegState G;

  const int tid = threadIdx.x, warp = tid >> 5;
  int lane;  // opaque: kept in a register instead of read again from the special register
  asm volatile("mov.u32 %0, %%laneid;" : "=r"(lane));
  WarpList<BLK>& W = lists[warp];
  const unsigned lt_mask = (1u << lane) - 1u;
  if (tid == 0) B.seg = first_segment(L);
  for (int k = tid; k < L.hist_width + 2 * kGuard; k += BLOCK) sh[k - kGuard] = 0u;
  __syncthreads();

  for (;;) {
    if (B.seg < 0) break;
    if (tid == 0) attach_segment(L, B, G);
    __syncthreads();
    if (tid < 27) {
      const Pos v = image_vector(*G.F, tid, G.grid);
      G.V4[tid] = make_float4(v.h.x, v.h.y, v.h.z, v.l.x);
      G.V2[tid] = make_float2(v.l.y, v.l.z);
    }
    __syncthreads();
    int qcount = 0;
    if (lane == 0) W.uni = W.axis = W.cull = 0ull;
    long long u = B.base + (long long)warp * B.len;
    int len = (int)min((long long)B.len, min(B.first - (long long)warp * B.len, G.items - u));

    for (;;) {
      if (len <= 0) {
        if (lane == 0) {
          const long long part = (G.items - *(volatile long long*)&B.seen) / G.claimers;
          len = (int)max(1LL, min(part, 1024LL));
          u = G.items ? (long long)atomicAdd(G.next, (unsigned long long)len) : 0LL;
          *(volatile long long*)&B.seen = u + len;
          len = (int)min((long long)len, G.items - u);
        }
        len = __shfl_sync(kFull, len, 0);
        u = __shfl_sync(kFull, u, 0);
        if (len <= 0) break;
      }

      unsigned listed = 0;
      int ri, rj, sub;
      item_of(G, u, ri, rj, sub);

      while (len > 0) {
        const int row = min(len, (G.n_tj - rj) * G.split - sub);
        len -= row;
        // ---- the run: state and factors
        const int i_begin = ri * kRun, ni = min(kRun, G.ni - i_begin), nj = G.nj;
        const int part = G.part;
        IRegs I;
        int pf = rj * kRun + sub * part;
        float4 pa = __ldg(G.P4j + min(pf + lane, nj - 1));
        float2 pb = __ldg(G.P2j + min(pf + lane, nj - 1));
        {
          const RunState R = run_state(G, __ldg(G.bi + 2 * ri), __ldg(G.bi + 2 * ri + 1));
          __syncwarp();
          if (lane == 0) W.R = R;
          __syncwarp();
          load_run(G, R.c, i_begin, ni, lane, I);
        }
        int tail = 0, done = 0;
        // the list's images: none near the run, every pair in the sweep
        bool near = G.all != 0, inner = true;
        for (int t = 0; t < row; ++t) {
          const bool diag = G.intra && rj == ri;
          const int jbeg = rj * kRun + sub * part;
          int jend = min(nj, jbeg + part);
          if (G.slow) {
            const int counted = slow_item(G, ri, rj, ni, jbeg, jend, sh, lane);
            if (counted >= 0) {
              listed += (unsigned)counted;
              jend = jbeg;  // nothing to list
            }
          }
          // ---- images of the j run that can lie in the sweep (bounds against bounds)
          bool keep = false;
          float g2 = 0.0f, f2 = 0.0f;
          if (lane < G.n_img && jbeg < jend) {
            const float4 jlo = __ldg(G.bj + 2 * rj), jhi = __ldg(G.bj + 2 * rj + 1);
            const int m = G.n_img == 1 ? kHome : lane;
            const float4 V = G.V4[m];
            const float sx = V.x, sy = V.y, sz = V.z;
            // ranges of the j run's image around the centre, then out by the half extents
            const float3 c = W.R.c, h = W.R.h;
            const float lx = jlo.x + sx - c.x, ux = jhi.x + sx - c.x;
            const float ly = jlo.y + sy - c.y, uy = jhi.y + sy - c.y;
            const float lz = jlo.z + sz - c.z, uz = jhi.z + sz - c.z;
            const float gx = fmaxf(fmaxf(lx, -ux) - h.x, 0.0f), gy = fmaxf(fmaxf(ly, -uy) - h.y, 0.0f),
                        gz = fmaxf(fmaxf(lz, -uz) - h.z, 0.0f);
            const float fx = fmaxf(fabsf(lx), fabsf(ux)) + h.x, fy = fmaxf(fabsf(ly), fabsf(uy)) + h.y,
                        fz = fmaxf(fabsf(lz), fabsf(uz)) + h.z;
            g2 = gx * gx + gy * gy + gz * gz;
            f2 = fx * fx + fy * fy + fz * fz;
            keep = g2 <= G.rc_hi2 && (PICK || f2 >= G.rc_lo2);
          }
          unsigned picked = 0u;  // PICK: several images, handled particle by particle
          if (PICK) {
            const bool img = lane < G.n_img && jbeg < jend;
            float far = img ? f2 : INFINITY;
            for (int o = 16; o > 0; o >>= 1) far = fminf(far, __shfl_xor_sync(kFull, far, o));
            // only images nearer than the farthest pair of another; none when one puts
            // every pair below the sweep
            const float reach = sqrtf(far) * (1.0f + 0x1p-15f) + 2.0f * G.abs;
            keep = keep && g2 <= reach * reach && far >= G.rc_lo2;
          }
          unsigned mask = __ballot_sync(kFull, keep);
          if (lane == 0) {  // statistics
            const unsigned long long np = (unsigned long long)max(jend - jbeg, 0) * (unsigned long long)ni;
            const int nimg = __popc(mask);
            if (nimg == 0) W.cull += np;
            if (nimg == 1) W.uni += np;
            if (nimg == 2) {
              const int a = __ffs(mask) - 1, b = 31 - __clz(mask);
              if ((a / 9 != b / 9) + (a / 3 % 3 != b / 3 % 3) + (a % 3 != b % 3) == 1) W.axis += np;
            }
          }
          // one round of 32 j particles of one image per turn; a last turn ends the
          // list with the row and with the diagonal item
          const bool ends = t == row - 1 || diag;
          int m = kHome, jb = jend;
          bool in_here = false, near_here = false;
          for (;;) {
            int want = BLK;
            if (PICK && jb >= jend && (mask & (mask - 1u))) {
              picked = mask;
              mask = 0u;
              in_here = inner = false;
              jb = jbeg;
            } else if (jb >= jend && mask) {
              const int ml = __ffs(mask) - 1;
              mask &= mask - 1u;
              picked = 0u;
              m = G.n_img == 1 ? kHome : ml;
              // inner: every pair in the sweep
              const float f2m = __shfl_sync(kFull, f2, ml), g2m = __shfl_sync(kFull, g2, ml);
              in_here = f2m <= G.in_hi2 && g2m >= G.in_lo2;
              inner = inner && in_here;
              const Pos o = image_origin(G, m, W.R.c);
              __syncwarp();
              if (lane == 0) W.o = o;
              __syncwarp();
              jb = jbeg;
            }
            const bool more = jb < jend;
            near_here = false;
            if (more) {
              const int jl = jb + lane;
              // this round's particle was loaded in the round before (the next
              // round, image or run is the likely successor); else load it now
              if (pf != jb) {
                pa = __ldg(G.P4j + min(jl, nj - 1));
                pb = __ldg(G.P2j + min(jl, nj - 1));
              }
              const Pos p = unpack(pa, pb);
              jb += 32;
              pf = jb < jend ? jb : (mask ? jbeg : jend);
              pa = __ldg(G.P4j + min(pf + lane, nj - 1));
              pb = __ldg(G.P2j + min(pf + lane, nj - 1));
              if constexpr (PICK) if (picked) {
                m = pick_round<MULTI>(G, W, picks[warp], picked, p, jl, jl < jend, i_begin, ni,
                                      diag ? i_begin : -(1 << 30), sh, lane, qcount);
                listed += 32u;  // (particles whose pairs it counted are not listed)
              }
              const float4 y =
                  j_image(p, PICK && picked ? image_origin(G, max(m, 0), W.R.c) : W.o, W.R.c1, W.R.c0);
              const float3 h = W.R.h;
              const float ax = fabsf(y.x), ay = fabsf(y.y), az = fabsf(y.z);
              const float gx = fmaxf(ax - h.x, 0.0f), gy = fmaxf(ay - h.y, 0.0f), gz = fmaxf(az - h.z, 0.0f);
              bool in = jl < jend && m >= 0 && gx * gx + gy * gy + gz * gz <= G.rc_hi2;
              if (MULTI) {  // (for a single image the same as below the sweep)
                const float fx = ax + h.x, fy = ay + h.y, fz = az + h.z;
                in = in && fx * fx + fy * fy + fz * fz >= G.rc_lo2;
              }
              const unsigned bal = __ballot_sync(kFull, in);
              // this round's own particles: near the run's box for their own W?
              const float w = __fmaf_rn(2.0f * W.R.c1, ax * ax + ay * ay + az * az, 2.0f * W.R.c0 + 3.0f + G.abs);
              near_here = __any_sync(kFull, in && gx * gx + gy * gy + gz * gz < w * w);
              near = near || near_here;
              if (in) {
                const int s = (tail + __popc(bal & lt_mask)) & (kCap - 1);
                float* a = reinterpret_cast<float*>(&W.A[s >> 1]) + (s & 1);
                float* b = reinterpret_cast<float*>(&W.B[s >> 1]) + (s & 1);
                a[0] = y.x;
                a[2] = y.y;
                b[0] = y.z;
                b[2] = y.w;
                W.ref[s] = (uint32_t)jl | ((uint32_t)m << kImgShift);
              }
              tail += __popc(bal);
            } else {
              if (!ends) break;
              want = (tail - done + 7) & ~7;  // fewer than a block: padded to whole groups
              if (want == 0) break;
              if (lane < done + want - tail) {
                const int s = (tail + lane) & (kCap - 1);
                reinterpret_cast<float*>(&W.B[s >> 1])[2 + (s & 1)] = NAN;
                W.ref[s] = 0u;
              }
            }
            __syncwarp();
            if (!more || tail - done >= BLK) {
              const int s0 = done & (kCap - 1);
              uint32_t groups, first = (uint32_t)i_begin;
              if (near || diag) {
                groups = list_near<MULTI>(G, W, i_begin, ni, s0, want, diag ? i_begin : -(1 << 30), sh, lane);
                first |= kNearPair;
              } else if (inner && more && ni == kRun && G.inner) {
                groups = list_block<INNER, MULTI>(G, I, W, s0, BLK, 0, sh, lane);
              } else {
                groups = list_block<PLAIN, MULTI>(G, I, W, s0, want, 0, sh, lane);
              }
              qcount = push_pairs(G, W, s0, groups, first, sh, lane, qcount);
              done += BLK;
              // what is left was appended in this round
              near = near_here || G.all;
              inner = !more || in_here;
            }
            if (!more) {
              listed += (unsigned)tail;
              tail = done = 0;
              break;
            }
          }
          if (++sub == G.split) {
            sub = 0;
            ++rj;
          }
        }
        if (rj == G.n_tj) {
          ++ri;
          rj = G.intra ? ri : 0;
        }
      }
      // flush before a shared count can pass 2^31: a warp that takes the total past a
      // multiple of kFlushPairs moves every word (the others keep counting)
      unsigned before = 0;
      if (lane == 0) before = atomicAdd(&B.since, listed);
      before = __shfl_sync(kFull, before, 0);
      if ((before ^ (before + listed)) >= kFlushPairs) {
        for (int k = lane; k < G.hi - G.lo; k += 32) merge_count(G.out + k, atomicExch(sh + k, 0u));
      }
    }
    // the first warp without items asks for the block's next segment
    if (lane == 0 && atomicExch(&B.asked, 1u) == 0u) B.next = own_segment(L);
    while (qcount > 0) qcount = list_drain(G, W.queue, qcount, sh, lane);
    if (lane == 0) {
      if (W.uni) atomicAdd(&G.F->uniform_pairs, W.uni);
      if (W.axis) atomicAdd(&G.F->axis_pairs, W.axis);
      if (W.cull) atomicAdd(&G.F->culled_pairs, W.cull);
    }

    __syncthreads();
    // ---- merge
    const int width = G.hi - G.lo;
    if (G.items) {
      uint64_t* const dst = G.out;
      for (int k = tid; k < width; k += BLOCK) {
        merge_count(dst + k, sh[k]);
        sh[k] = 0u;
      }
      for (int k = tid; k < 2 * kGuard; k += BLOCK) sh[k < kGuard ? k - kGuard : width + k - kGuard] = 0u;
    }
    next_segment(L, B, G, tid, lane);
  }
}

// ------------------------------------------------------------------ self check

// Sampled pairs of a frame (a block takes segment after segment of it) with the pair
// loop's arithmetic for their shortest image, against the binary64 definition: out[0] =
// largest |q - t64^2| / W over pairs inside the sweep (below 1), out[1] = pairs whose
// bin, as decided in float32 or by the double-float tier, is another (0), out[2] = pairs.
__device__ void check_listed_pair(const SegState& G, int i, int j, int lane, double* worst, unsigned long long* viol,
                                  unsigned long long* checked) {
  const FrameDev& F = *G.F;
  const int m = F.variant == V_NONE ? kHome : picked_image(F, G.i0 + i, G.j0 + j);
  if (m < 0) return;  // two images within rounding: re-decided in binary64
  const RunState R = run_state(G, __ldg(G.bi + 2 * (i / kRun)), __ldg(G.bi + 2 * (i / kRun) + 1));
  const float4 x = run_factor(G, i, i + 1, R.c);
  const float4 y = j_image(unpack(__ldg(G.P4j + j), __ldg(G.P2j + j)), image_origin(G, m, R.c), R.c1, R.c0);
  const float nq = __fadd_rn(__fmaf_rn(y.x, x.x, __fmaf_rn(y.y, x.y, __fmaf_rn(y.z, x.z, x.w))), y.w);
  const float w2 = __fmaf_rn(y.w, -2.0f * R.c1 * (1.0f + 0x1p-10f), 2.0f * R.c0 * (1.0f + 0x1p-10f));
  const double3 pi = coords64(F, G.i0 + i), pj = coords64(F, G.j0 + j);
  const double r2 = F.variant == V_NONE    ? exact_r2<V_NONE>(F, pi, pj)
                    : F.variant == V_ORTHO ? exact_r2<V_ORTHO>(F, pi, pj)
                    : F.variant == V_TRIC ? exact_r2<V_TRIC>(F, pi, pj)
                                          : exact_r2<V_TRIC_SEARCH>(F, pi, pj);
  const int k64 = bin_from_thresholds(F.T, F.S, F.nbins, r2);
  const double t64 = sqrt(r2) * ((double)F.nbins / F.r_max);
  if (t64 >= (double)G.lo && t64 < (double)G.hi) {
    *worst = fmax(*worst, fabs(0.5 * (double)w2 - (double)nq - t64 * t64) / (0.5 * (double)w2));
    ++*checked;
  }
  float sc = fminf(sqrt_approx(-nq), (float)(G.hi + 1 + lane));
  if (G.lo > 0) sc = fmaxf(sc, (float)(G.lo - lane));
  const float sm = __fadd_rn(sc, kMagicRound), n = __fadd_rn(sm, -kMagicRound), e = __fmaf_rn(n, n, nq);
  int bin;
  if (G.all || -nq < (w2 + 1.0f) * (w2 + 1.0f) || __float_as_uint(e) < __float_as_uint(w2)) {
    float edge;
    unsigned nexact = 0;
    bin = listed_bin(G, i, j, m, edge, nexact);
  } else {
    bin = G.lo + (__float_as_int(sm) + (int)(__float_as_uint(e) >> 31) - (__float_as_int(kMagicRound) + G.lo + 1));
  }
  const bool in = bin >= G.lo && bin < G.hi, in64 = k64 >= G.lo && k64 < G.hi;
  if (in != in64 || (in && bin != k64)) ++*viol;
}

__global__ void check_list_kernel(const ListSegment* segs, int n_segs, uint64_t n_samples, uint64_t seed,
                                  unsigned long long* out) {
  __shared__ SegState G;
  const int tid = threadIdx.x, lane = tid & 31;
  double worst = 0.0;
  unsigned long long viol = 0, checked = 0;
  const uint64_t each = (n_samples + n_segs - 1) / n_segs;
  for (int seg = 0; seg < n_segs; ++seg) {
    __syncthreads();
    if (tid == 0) enter_segment(segs[seg], G);
    __syncthreads();
    if (tid < 27) {
      const Pos v = image_vector(*G.F, tid, G.grid);
      G.V4[tid] = make_float4(v.h.x, v.h.y, v.h.z, v.l.x);
      G.V2[tid] = make_float2(v.l.y, v.l.z);
    }
    __syncthreads();
    if (G.slow || G.items == 0) continue;  // (binary64)
    for (uint64_t s = blockIdx.x * (uint64_t)blockDim.x + tid; s < each; s += (uint64_t)gridDim.x * blockDim.x) {
      uint64_t h = (seed + s + (uint64_t)seg * each) * 0x9E3779B97F4A7C15ull;
      h = (h ^ (h >> 30)) * 0xBF58476D1CE4E5B9ull;
      h = (h ^ (h >> 27)) * 0x94D049BB133111EBull;
      h ^= h >> 31;
      const int i = (int)(h % (uint64_t)G.ni), j = (int)((h >> 32) % (uint64_t)G.nj);
      if (G.intra && i == j) continue;
      check_listed_pair(G, i, j, lane, &worst, &viol, &checked);
    }
  }
  for (int o = 16; o > 0; o >>= 1) {
    worst = fmax(worst, __shfl_xor_sync(kFull, worst, o));
    viol += __shfl_xor_sync(kFull, viol, o);
    checked += __shfl_xor_sync(kFull, checked, o);
  }
  if (lane == 0) {
    atomicMax(out, (unsigned long long)__double_as_longlong(worst));
    atomicAdd(out + 1, viol);
    atomicAdd(out + 2, checked);
  }
}

size_t smem_of(size_t list_bytes, int hist_width) {
  return list_bytes * (kListBlock / 32) + 4 * ((size_t)hist_width + 2 * kGuard);
}

// Dynamic shared memory per block: the device's, less the kernel's static part.
size_t smem_limit() {
  int dev = 0, optin = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  return (size_t)std::max(optin - 1024, 0);
}

template <bool MULTI, bool PICK, int BLK>
cudaError_t launch_list_t(const ListLaunch& p, int grid, cudaStream_t stream) {
  const size_t smem = smem_of(sizeof(WarpList<BLK>) + (PICK ? sizeof(PickList) : 0), p.hist_width);
  cudaError_t e =
      cudaFuncSetAttribute(list_kernel<MULTI, PICK, BLK>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  list_kernel<MULTI, PICK, BLK><<<grid, kListBlock, smem, stream>>>(p);
  return cudaGetLastError();
}

}  // namespace

int list_kernel_max_width() {
  const size_t limit = smem_limit(), fixed = smem_of(sizeof(WarpList<kBlkNarrow>), 0);
  return limit <= fixed ? 0 : (int)((limit - fixed) / 4) & ~3;
}

cudaError_t launch_check_list(const ListSegment* segs, int n_segs, uint64_t n_samples, uint64_t seed,
                              unsigned long long* out, cudaStream_t stream) {
  (void)cudaGetLastError();
  if (n_segs <= 0) return cudaSuccess;
  check_list_kernel<<<1024, 256, 0, stream>>>(segs, n_segs, n_samples, seed, out);
  return cudaGetLastError();
}

// Blocks of 64 images where the histogram leaves room for their lists, else of 32,
// which cost 2 % (N = 1,000,000 orthorhombic 172 -> 176 ms) and save a sweep: no box,
// N = 100,000, 45,000 bins 3.72 ms in two sweeps, 2.99 in one.
cudaError_t launch_list(const ListLaunch& p, int grid, cudaStream_t stream) {
  (void)cudaGetLastError();
  if (p.pick)
    return p.multi ? launch_list_t<true, true, kBlk>(p, grid, stream) : launch_list_t<false, true, kBlk>(p, grid, stream);
  if (smem_of(sizeof(WarpList<kBlk>), p.hist_width) <= smem_limit())
    return p.multi ? launch_list_t<true, false, kBlk>(p, grid, stream) : launch_list_t<false, false, kBlk>(p, grid, stream);
  return p.multi ? launch_list_t<true, false, kBlkNarrow>(p, grid, stream)
                 : launch_list_t<false, false, kBlkNarrow>(p, grid, stream);
}

}  // namespace dh
