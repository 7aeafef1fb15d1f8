// CUDA kernels of the particle-pair distance histogram (sm_103a).
//
// Hot path (Reuter & Koefinger, Sec. 2 and 3.2): for every unique pair the
// distance vector, the minimum image of Eq. 5, the Euclidean distance and the
// bin kappa = (int) nbins r / r_max of Alg. 1 are computed, and the bin of a
// block-private shared-memory histogram is incremented (the hybrid strategy of
// Sec. 2.4: groups of threads share a private histogram, merged into the
// global one at the end, Sec. 3.2.3).  Private counts are uint32 and are
// flushed into the uint64 global histogram before they can overflow
// (Sec. 3.1, also applied on the GPU).
//
// Precision design (not in the paper, which computes in float32 only): the
// result must equal the binary64 definition bin for bin.  Each pair is first
// evaluated in float32 with an error bound delta (in bin units) derived for the
// exact operation sequence below; a pair whose float32 bin coordinate t lies
// farther than delta from every integer is decided in float32.  The others are
// pushed into a per-warp queue and re-decided by replaying the binary64
// definition (same operations, same order, explicit round-to-nearest
// intrinsics, no contraction) and comparing r^2 with a table of binary64
// thresholds T[k] = smallest r^2 whose bin is >= k.
#include <cooperative_groups.h>
#include <float.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>
#include <cmath>

#include "dh_device.h"
#include "dh_internal.h"

namespace dh {

// ------------------------------------------------------------------ helpers

// Every launcher reports the error of its own launch: a non-sticky error that an
// earlier, unrelated API call on this thread left behind (this library's or
// another's) is cleared first.  Errors of kernels already running are sticky
// and still surface at the next synchronisation.
static inline void clear_stale_error() { (void)cudaGetLastError(); }

// ------------------------------------------------------------------ binary64 bin of Alg. 1

// kappa = floor((nbins * sqrt(r2)) / r_max), evaluated left to right in
// binary64; nbins when the pair is beyond the histogram.
__host__ __device__ inline int64_t bin_of_b64(double r2, double r_max, int32_t nbins) {
#ifdef __CUDA_ARCH__
  double r = __dsqrt_rn(r2);
  double t = __dmul_rn((double)nbins, r);
  t = __ddiv_rn(t, r_max);
#else
  double r = std::sqrt(r2);
  double t = (double)nbins * r;
  t = t / r_max;
#endif
  if (!(t < (double)nbins)) return nbins;
  return (int64_t)floor(t);
}

// Smallest binary64 q >= 0 with bin(q) >= k (k >= 1), found by stepping ulp by
// ulp from the rounded edge (k r_max / nbins)^2.  *ok is cleared if the walk
// does not settle within 4096 steps.
__host__ __device__ inline double threshold_of(int32_t k, double r_max, int32_t nbins, int* ok) {
  if (k <= 0) return 0.0;
  double e = ((double)k * r_max) / (double)nbins;
  double q = e * e;
  int it = 0;
  if (bin_of_b64(q, r_max, nbins) >= k) {
    for (; it < 4096; ++it) {
      double p = nextafter(q, 0.0);
      if (!(p < q) || bin_of_b64(p, r_max, nbins) < k) break;
      q = p;
    }
  } else {
    for (; it < 4096; ++it) {
      q = nextafter(q, (double)INFINITY);
      if (bin_of_b64(q, r_max, nbins) >= k) break;
    }
  }
  if (it >= 4096) *ok = 0;
  return q;
}

int64_t host_bin_of(double r2, double r_max, int32_t nbins) { return bin_of_b64(r2, r_max, nbins); }

int build_thresholds_host(double r_max, int32_t nbins, double* T) {
  int ok = 1;
  for (int32_t k = 0; k <= nbins; ++k) T[k] = threshold_of(k, r_max, nbins, &ok);
  return ok;
}

// T[k] for k = 0..nbins, followed by the same values as float pairs (hi, lo)
// at (float2*)(T + nbins + 1) for the double-float tier.
__global__ void thresholds_kernel(double r_max, int32_t nbins, double* T, int32_t* status) {
  int32_t k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k > nbins) return;
  int ok = 1;
  double t = threshold_of(k, r_max, nbins, &ok);
  T[k] = t;
  float hi = __double2float_rn(t);
  float lo = __double2float_rn(t - (double)hi);
  reinterpret_cast<float2*>(T + nbins + 1)[k] = make_float2(hi, lo);
  if (!ok) atomicExch(status, 7);
}

// ------------------------------------------------------------------ A1: staging

// Fractional coordinates in float32 (triclinic; orthorhombic too).
__device__ __forceinline__ float3 frac_coords(const FrameDev& F, float x, float y, float z) {
  const float s2 = z * F.invf[2];
  const float s1 = (y - F.Bf[5] * s2) * F.invf[1];
  return make_float3((x - F.Bf[1] * s1 - F.Bf[2] * s2) * F.invf[0], s1, s2);
}

// Staging of several frames at once: block b handles chunk b of the job whose
// chunk range contains it; coords (n x stride floats, or doubles) -> float4
// (and double4 for binary64 input), per-axis min/max of the float32 values (for
// the error window) and finiteness.
__global__ void stage_kernel(const StageJob* __restrict__ jobs, int n_jobs) {
  const long long chunk = blockIdx.x;
  int lo = 0, hi = n_jobs - 1;
  while (lo < hi) {
    int mid = (lo + hi + 1) >> 1;
    if (jobs[mid].chunk0 <= chunk) lo = mid; else hi = mid - 1;
  }
  const StageJob J = jobs[lo];
  const int64_t i0 = (chunk - J.chunk0) * (int64_t)kStageChunk;
  const int64_t i1 = min(J.n, i0 + (int64_t)kStageChunk);
  float mn0 = INFINITY, mn1 = INFINITY, mn2 = INFINITY;
  float mx0 = -INFINITY, mx1 = -INFINITY, mx2 = -INFINITY;
  // triclinic: the range of the fractional coordinates too (does the frame span more than one cell?)
  const bool frac = J.fd->variant == V_TRIC || J.fd->variant == V_TRIC_SEARCH;
  float sn[3] = {INFINITY, INFINITY, INFINITY}, sx[3] = {-INFINITY, -INFINITY, -INFINITY};
  int bad = 0;
  const float* __restrict__ src = J.src;
  const int stride = J.stride;
  const double* __restrict__ src64 = reinterpret_cast<const double*>(src);
  for (int64_t i = i0 + threadIdx.x; i < i1; i += blockDim.x) {
    float x, y, z;
    if (J.dst64) {  // binary64 input: kept as given, and rounded to float32 for the fast path
      double a = src64[i * stride], b = src64[i * stride + 1], c = src64[i * stride + 2];
      J.dst64[i] = make_double4(a, b, c, 0.0);
      x = __double2float_rn(a);
      y = __double2float_rn(b);
      z = __double2float_rn(c);
    } else {
      x = src[i * stride];
      y = src[i * stride + 1];
      z = src[i * stride + 2];
    }
    bad |= !(isfinite(x) && isfinite(y) && isfinite(z));
    J.dst[i] = make_float4(x, y, z, 0.0f);
    mn0 = fminf(mn0, x); mn1 = fminf(mn1, y); mn2 = fminf(mn2, z);
    mx0 = fmaxf(mx0, x); mx1 = fmaxf(mx1, y); mx2 = fmaxf(mx2, z);
    if (frac) {
      const float3 s = frac_coords(*J.fd, x, y, z);
      sn[0] = fminf(sn[0], s.x); sn[1] = fminf(sn[1], s.y); sn[2] = fminf(sn[2], s.z);
      sx[0] = fmaxf(sx[0], s.x); sx[1] = fmaxf(sx[1], s.y); sx[2] = fmaxf(sx[2], s.z);
    }
  }
  // block minima and maxima (maxima as minima of the negated values), one set of
  // atomics per block
  float v[12] = {mn0, mn1, mn2, -mx0, -mx1, -mx2, sn[0], sn[1], sn[2], -sx[0], -sx[1], -sx[2]};
  __shared__ float s_v[8][12];
  __shared__ int s_bad;
  if (threadIdx.x == 0) s_bad = 0;
  __syncthreads();
  const int nv = frac ? 12 : 6;
#pragma unroll
  for (int c = 0; c < 12; ++c) {
    if (c >= nv) break;
    for (int o = 16; o > 0; o >>= 1) v[c] = fminf(v[c], __shfl_xor_sync(kFull, v[c], o));
    if ((threadIdx.x & 31) == 0) s_v[threadIdx.x >> 5][c] = v[c];
  }
  if (bad) s_bad = 1;
  __syncthreads();
  if (threadIdx.x < nv) {
    const int c = threadIdx.x;
    float m = s_v[0][c];
    for (int w = 1; w < blockDim.x / 32; ++w) m = fminf(m, s_v[w][c]);
    FrameDev* F = J.fd;
    int32_t* const mn = c < 6 ? F->cmin : F->smin;
    int32_t* const mx = c < 6 ? F->cmax : F->smax;
    if (c % 6 < 3) {
      if (m < INFINITY) atomicMin(mn + c % 3, ord_of(m));
    } else if (m < INFINITY) {
      atomicMax(mx + c % 3, ord_of(-m));
    }
  }
  if (threadIdx.x == 0 && s_bad) atomicExch(&J.fd->bad, 1);
}

// ------------------------------------------------------------------ spatial order (staging)

// Position of cell (x, y, z) of a 2^g grid along the three-dimensional Hilbert
// curve, by J. Skilling's transpose algorithm (AIP Conf. Proc. 707, 381, 2004).
// Unlike Morton order its consecutive cells are always neighbours, so runs of
// consecutive particles have smaller bounding boxes.
__device__ __forceinline__ uint32_t hilbert_key(uint32_t x, uint32_t y, uint32_t z, int g) {
  for (uint32_t q = 1u << (g - 1); q > 1; q >>= 1) {  // undo the excess work, axis by axis
    const uint32_t p = q - 1;
    if (x & q) x ^= p;
    if (y & q) {
      x ^= p;
    } else {
      const uint32_t t = (x ^ y) & p;
      x ^= t;
      y ^= t;
    }
    if (z & q) {
      x ^= p;
    } else {
      const uint32_t t = (x ^ z) & p;
      x ^= t;
      z ^= t;
    }
  }
  y ^= x;  // Gray encoding
  z ^= y;
  uint32_t t = 0;
  for (uint32_t q = 1u << (g - 1); q > 1; q >>= 1)
    if (z & q) t ^= q - 1;
  x ^= t;
  y ^= t;
  z ^= t;
  uint32_t key = 0;
  for (int b = g - 1; b >= 0; --b) key = (key << 3) | (((x >> b) & 1u) << 2) | (((y >> b) & 1u) << 1) | ((z >> b) & 1u);
  return key;
}

// A particle's position brought home: minus the lattice vector of its fractional
// coordinates' integer parts (frames that span several cells). In binary64, of
// which the SM does two operations per cycle,
__device__ __forceinline__ double3 bring_home(const FrameDev& F, double x, double y, double z) {
  const double* B = F.B;
  const double sz = z / B[8], sy = (y - B[5] * sz) / B[4], sx = (x - B[1] * sy - B[2] * sz) / B[0];
  const double kx = floor(sx), ky = floor(sy), kz = floor(sz);
  return make_double3(((x - kx * B[0]) - ky * B[1]) - kz * B[2], (y - ky * B[4]) - kz * B[5], z - kz * B[8]);
}

// or in double-floats: the second turn removes what the first one's float32
// quotients left (they err by a fraction of a cell up to 2^20 cells).  The
// subtractions err by less than 2^-44 of the coordinates (list_setup).
struct DF3 {
  DF x, y, z;
};
__device__ __noinline__ DF3 bring_home_df(const FrameDev& F, float x, float y, float z) {
  DF3 v{{x, 0.0f}, {y, 0.0f}, {z, 0.0f}};
  for (int turn = 0; turn < 2; ++turn) {
    const float3 s = frac_coords(F, v.x.h, v.y.h, v.z.h);
    const float kx = floorf(s.x), ky = floorf(s.y), kz = floorf(s.z);
    v.x = df_sub_kb(df_sub_kb(df_sub_kb(v.x, kx, F.Bf[0], F.Bl[0]), ky, F.Bf[1], F.Bl[1]), kz, F.Bf[2], F.Bl[2]);
    v.y = df_sub_kb(df_sub_kb(v.y, ky, F.Bf[4], F.Bl[4]), kz, F.Bf[5], F.Bl[5]);
    v.z = df_sub_kb(v.z, kz, F.Bf[8], F.Bl[8]);
  }
  return v;
}
__device__ __forceinline__ float3 home32(const FrameDev& F, float x, float y, float z) {
  if (F.wrap == 1) {
    const DF3 v = bring_home_df(F, x, y, z);
    return make_float3(v.x.h, v.y.h, v.z.h);
  }
  const double3 w = bring_home(F, x, y, z);
  return make_float3((float)w.x, (float)w.y, (float)w.z);
}

// Bins beyond which a far coordinate is moved in to, so that sums of squares stay
// finite.  Differences only get smaller by it: bounds of such runs remain lower bounds.
constexpr float kFarthest = 0x1p60f;

// One coordinate in bins: its high part on the grid, and the rest.
__device__ __forceinline__ DF to_bins_on_grid(const FrameDev& F, DF v) {
  const DF p = two_prod(v.h, F.S);
  if (fabsf(p.h) >= F.list_far) return {fminf(fmaxf(p.h, -kFarthest), kFarthest), 0.0f};
  const DF s = two_sum(p.h, __fmaf_rn(v.h, F.S_l, __fmaf_rn(v.l, F.S, p.l)));
  const float h = on_grid(s.h, F.list_grid);
  return {h, __fadd_rn(__fsub_rn(s.h, h), s.l)};
}
// The list kernel's position of a particle (x64: its binary64 input, if it has one).
__device__ __forceinline__ void list_position(const FrameDev& F, float4 p, const double4* x64, float4& P4, float2& P2) {
  DF x, y, z;
  if (x64 || F.wrap == 2) {
    double3 v = x64 ? make_double3(x64->x, x64->y, x64->z) : make_double3(p.x, p.y, p.z);
    if (F.wrap) v = bring_home(F, v.x, v.y, v.z);
    const double s = (double)F.S + (double)F.S_l;
    double3 t = make_double3(v.x * s, v.y * s, v.z * s);
    if (F.list_far < INFINITY) {
      t.x = fmin(fmax(t.x, -(double)kFarthest), (double)kFarthest);
      t.y = fmin(fmax(t.y, -(double)kFarthest), (double)kFarthest);
      t.z = fmin(fmax(t.z, -(double)kFarthest), (double)kFarthest);
    }
    x.h = on_grid((float)t.x, F.list_grid);
    y.h = on_grid((float)t.y, F.list_grid);
    z.h = on_grid((float)t.z, F.list_grid);
    x.l = (float)(t.x - (double)x.h);
    y.l = (float)(t.y - (double)y.h);
    z.l = (float)(t.z - (double)z.h);
  } else {
    DF3 v{{p.x, 0.0f}, {p.y, 0.0f}, {p.z, 0.0f}};
    if (F.wrap) v = bring_home_df(F, p.x, p.y, p.z);
    x = to_bins_on_grid(F, v.x);
    y = to_bins_on_grid(F, v.y);
    z = to_bins_on_grid(F, v.z);
  }
  P4 = make_float4(x.h, y.h, z.h, x.l);
  P2 = make_float2(y.l, z.l);
}

// Cell of a particle in a pass of the spatial order (only the order depends on it):
// on the curve, or its slab's (pass 1) or column's (pass 2) cell along the pass's
// axis.  rank: its place after the pass before.
__device__ __forceinline__ int sort_cell(const FrameDev& F, const SortSeg& S, float4 p, int pass, int rank) {
  if (S.nb[0] == 0 && S.g == 0) return 0;
  if (F.wrap) {
    const float3 w = home32(F, p.x, p.y, p.z);
    p.x = w.x;
    p.y = w.y;
    p.z = w.z;
  }
  if (S.nb[0]) {
    const int nb = S.nb[pass];
    const float v = pass == 0 ? p.x - F.key_lo[0] : pass == 1 ? p.y - F.key_lo[1] : p.z - F.key_lo[2];
    int group = 0;
    if (pass > 0) group = rank / S.slab;
    if (pass > 1) group = group * S.n_col + (rank - group * S.slab) / S.col;
    return group * nb + min(max((int)(v * F.key_inv * (float)nb), 0), nb - 1);
  }
  const float G = (float)(1 << S.g);
  const int last = (1 << S.g) - 1;
  const int cx = (int)((p.x - F.key_lo[0]) * F.key_inv * G), cy = (int)((p.y - F.key_lo[1]) * F.key_inv * G),
            cz = (int)((p.z - F.key_lo[2]) * F.key_inv * G);
  return (int)hilbert_key((uint32_t)min(max(cx, 0), last), (uint32_t)min(max(cy, 0), last),
                          (uint32_t)min(max(cz, 0), last), S.g);
}

// The segment of this block: the last whose first block (first(segment)) is not above it.
template <typename First>
__device__ __forceinline__ const SortSeg& segment_of_block(const SortSeg* segs, int n_segs, First first) {
  int lo = 0, hi = n_segs - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (first(segs[mid]) <= (int)blockIdx.x) lo = mid; else hi = mid - 1;
  }
  return segs[lo];
}

// One pass: each particle's cell and its place in the cell (keys), the cells' counts.
__global__ void sort_count_kernel(const SortSeg* segs, int n_segs, int pass, const float4* __restrict__ X, int2* keys,
                                  uint32_t* counts, const uint32_t* __restrict__ cursors) {
  const SortSeg S = segment_of_block(segs, n_segs, [](const SortSeg& s) { return s.chunk0; });
  if (pass < 2 && S.nb[0] == 0) return;
  const int64_t i0 = (int64_t)((int)blockIdx.x - S.chunk0) * kSortChunk;
  const int64_t i1 = min((int64_t)S.n, i0 + kSortChunk);
  for (int64_t i = i0 + threadIdx.x; i < i1; i += blockDim.x) {
    int rank = 0;
    if (pass > 0 && S.nb[0]) {
      const int2 k = keys[S.x0 + i];
      rank = (int)cursors[S.key0[pass - 1] + k.x] + k.y;
    }
    const int cell = sort_cell(*S.fd, S, X[S.x0 + i], pass, rank);
    keys[S.x0 + i] = make_int2(cell, (int)atomicAdd(counts + S.key0[pass] + cell, 1u));
  }
}

// Exclusive prefix sum of each segment's counters (counts -> cursors), one block
// per kScanTile of them.  A block sums the counters before its tile itself, from L2
// in 16-byte loads: up to 6 MB at N = 1,000,000 (1.5 counters a particle, 1.1 GB over
// all blocks), cheaper than a second launch or a wait on the blocks before it (a single
// block per segment took 0.42 ms at 2^18 counters, one tenth of what the whole frame's
// other preparation took).  The sum grows with the square of the counters: at N = 10^7
// 60 MB a block and 110 GB over all of them, from where on a second level would pay.
__global__ void __launch_bounds__(1024) sort_scan_kernel(const SortSeg* segs, int n_segs, int pass,
                                                         const uint32_t* __restrict__ counts,
                                                         uint32_t* __restrict__ cursors) {
  const SortSeg S = segment_of_block(segs, n_segs, [pass](const SortSeg& s) { return s.tile0[pass]; });
  const int m = (int)sort_keys(S, pass), t0 = ((int)blockIdx.x - S.tile0[pass]) * kScanTile;
  if (t0 >= m) return;
  const uint32_t* c = counts + S.key0[pass];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  __shared__ uint32_t s_sum[32];
  // this thread's four counters (segments below four counters have a whole tile to themselves)
  uint32_t v[4], local = 0;
  for (int q = 0; q < 4; ++q) {
    const int k = t0 + 4 * tid + q;
    v[q] = k < m ? c[k] : 0u;
    local += v[q];
  }
  // counters before the tile (a multiple of four, 16-byte aligned: see key0)
  uint32_t before = 0;
  const uint4* c4 = reinterpret_cast<const uint4*>(c);
#pragma unroll 4
  for (int k = tid; k < t0 / 4; k += 1024) {
    const uint4 x = __ldg(c4 + k);
    before += (x.x + x.y) + (x.z + x.w);
  }
  for (int o = 16; o > 0; o >>= 1) before += __shfl_xor_sync(kFull, before, o);
  if (lane == 0) s_sum[warp] = before;
  __syncthreads();
  uint32_t base = s_sum[lane];
  for (int o = 16; o > 0; o >>= 1) base += __shfl_xor_sync(kFull, base, o);
  __syncthreads();
  uint32_t incl = local;
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t x = __shfl_up_sync(kFull, incl, o);
    if (lane >= o) incl += x;
  }
  if (lane == 31) s_sum[warp] = incl;
  __syncthreads();
  uint32_t w = lane < warp ? s_sum[lane] : 0u;
  for (int o = 16; o > 0; o >>= 1) w += __shfl_xor_sync(kFull, w, o);
  uint32_t run = base + w + incl - local;
  for (int q = 0; q < 4; ++q) {
    const int k = t0 + 4 * tid + q;
    if (k < m) cursors[S.key0[pass] + k] = run;
    run += v[q];
  }
}

__global__ void sort_scatter_kernel(const SortSeg* segs, int n_segs, const float4* __restrict__ src,
                                    const double4* __restrict__ src64, const int2* __restrict__ keys,
                                    const uint32_t* __restrict__ cursors, float4* dst, double4* dst64) {
  const SortSeg S = segment_of_block(segs, n_segs, [](const SortSeg& s) { return s.chunk0; });
  const FrameDev& F = *S.fd;
  const int64_t i0 = (int64_t)((int)blockIdx.x - S.chunk0) * kSortChunk;
  const int64_t i1 = min((int64_t)S.n, i0 + kSortChunk);
  for (int64_t i = i0 + threadIdx.x; i < i1; i += blockDim.x) {
    const int2 k = keys[S.x0 + i];
    const int64_t pos = S.x0 + cursors[S.key0[2] + k.x] + k.y;
    const float4 p = src[S.x0 + i];
    dst[pos] = p;
    double4 q;
    if (F.X64) dst64[pos] = q = src64[S.x0 + i];
    if (F.P4) list_position(F, p, F.X64 ? &q : nullptr, F.P4[pos - S.f0], F.P2[pos - S.f0]);
  }
}

// Bounds of one run of kRun ordered particles (by one warp), over the positions
// the list kernel works with.
__device__ __forceinline__ void run_bounds(const FrameDev& F, const SortSeg& S, int run, int lane) {
  float b[6] = {INFINITY, INFINITY, INFINITY, -INFINITY, -INFINITY, -INFINITY};
  const int64_t p0 = S.x0 - S.f0;
  for (int i = run * kRun + lane; i < min(S.n, (run + 1) * kRun); i += 32) {
    const float4 p = __ldcg(F.P4 + p0 + i);
    const float v[3] = {p.x, p.y, p.z};
    for (int c = 0; c < 3; ++c) {
      b[c] = fminf(b[c], v[c]);
      b[3 + c] = fmaxf(b[3 + c], v[c]);
    }
  }
  for (int o = 16; o > 0; o >>= 1)
    for (int c = 0; c < 3; ++c) {
      b[c] = fminf(b[c], __shfl_xor_sync(kFull, b[c], o));
      b[3 + c] = fmaxf(b[3 + c], __shfl_xor_sync(kFull, b[3 + c], o));
    }
  if (lane == 0) {
    const float most = fmaxf(fmaxf(fmaxf(-b[0], b[3]), fmaxf(-b[1], b[4])), fmaxf(-b[2], b[5]));
    F.bnd[2 * (S.run0 + run)] = make_float4(b[0], b[1], b[2], most >= F.list_far ? 1.0f : 0.0f);
    F.bnd[2 * (S.run0 + run) + 1] = make_float4(b[3], b[4], b[5], 0.0f);
  }
}
__global__ void run_bounds_kernel(const SortSeg* segs, int n_segs) {
  const SortSeg S = segment_of_block(segs, n_segs, [](const SortSeg& s) { return s.bblock0; });
  const int run = ((int)blockIdx.x - S.bblock0) * kBoundRuns + threadIdx.x / 32;
  if (S.fd->bnd && run * (int64_t)kRun < S.n) run_bounds(*S.fd, S, run, threadIdx.x & 31);
}

// ------------------------------------------------------------------ per-frame error window

// Largest rounding error (half an ulp) of a float32 result whose exact value
// has magnitude at most D.
__device__ inline double half_ulp_below(double D) {
  if (!(D > 0.0)) return 0.0;
  int E;
  frexp(D, &E);  // D = m 2^E, m in [1/2, 1): |x| <= D < 2^E
  return ldexp(1.0, E - 25);
}

// No box, one sweep: the largest distance D maps below nbins + 1 even after the
// float32 roundings of q and of its square root (relative 2^-18 covers them).
__device__ __forceinline__ bool inside_one_sweep(const FrameDev& F, double D) {
  return F.variant == V_NONE && F.sweep_width >= F.nbins &&
         ((double)F.S + (double)F.S_l) * D * (1.0 + 1.0 / 262144.0) < (double)F.nbins + 1.0;
}

// The spatial order's grid and the list kernel's window of one frame.
//
// The list kernel works in bins, relative to the centre of an i run: x for the
// run's particles (|x| <= H, half the diagonal of its bounds), y for an image of
// a j particle (T = |y|), both double-floats, and evaluates
//   q = A + (B - 2 x.y),  A = |y|^2, B = |x|^2,
// A and B rounded once, x and y rounded once for the product, the parenthesis
// first (three FMAs), A added last.  With u = 2^-24, q errs by at most
//   x and y rounded for the product         2u TH + 2u TH
//   A, B                                    u T^2 + u H^2
//   three FMAs, results below 2 TH + H^2    6u TH + 3u H^2
//   last add                                u (T + H)^2
// in all u (2 T^2 + 12 TH + 5 H^2) <= u ((2 + 6l) T^2 + (5 + 6/l) H^2) for any
// l > 0 (run_state takes l = H over a typical T).  list_c0 covers what the
// double-floats leave out (a0: positions, 2^-47 each and per axis, the products
// with S and the image vectors) and the binary64 definition's own rounding of t.
__device__ void list_setup(FrameDev& F, const double* R, const double* Xm) {
  const double u = 1.0 / 16777216.0;
  const double* B = F.B;
  const double S = (double)F.S + (double)F.S_l;
  int wrap = 0, slow = 0;
  double lo[3], ext[3], far = 0.0;
  for (int c = 0; c < 3; ++c) {
    lo[c] = (F.cmin[c] <= F.cmax[c]) ? (double)float_of_ord(F.cmin[c]) : 0.0;
    ext[c] = R[c];
    far = fmax(far, Xm[c]);
  }
  if (F.variant != V_NONE) {
    // What the span may be off by, in cells: binary64 input was rounded to float32 at both
    // ends, and the fractional coordinates of a triclinic cell come from a chain of less
    // than 14 roundings of magnitudes up to the coordinates'.
    double off[3] = {0.0, 0.0, 0.0};
    if (F.X64 || F.variant != V_ORTHO) {
      const double per = F.variant != V_ORTHO ? 32.0 * u : 0.0;
      double e[3];
      for (int c = 0; c < 3; ++c) e[c] = per * Xm[c] + (F.X64 ? 2.0 * half_ulp_below(Xm[c]) : 0.0);
      off[2] = e[2] * (double)F.invf[2];
      off[1] = (e[1] + fabs(B[5]) * off[2]) * (double)F.invf[1];
      off[0] = (e[0] + fabs(B[1]) * off[1] + fabs(B[2]) * off[2]) * (double)F.invf[0];
    }
    for (int c = 0; c < 3; ++c) {
      const double span = F.variant != V_ORTHO ? (double)float_of_ord(F.smax[c]) - (double)float_of_ord(F.smin[c])
                                               : R[c] * (double)F.invf[c];
      // with the search, the nearest image can differ by nearly a cell more (check_frame)
      if (!(span + off[c] <= 1.0 + (F.variant == V_TRIC_SEARCH ? 1.0 / 16384.0 : 1.0 / 16.0))) wrap = 1;
    }
    if (wrap) {  // the home cell's bounding box
      ext[0] = B[0] + fabs(B[1]) + fabs(B[2]);
      ext[1] = B[4] + fabs(B[5]);
      ext[2] = B[8];
      lo[0] = fmin(B[1], 0.0) + fmin(B[2], 0.0);
      lo[1] = fmin(B[5], 0.0);
      lo[2] = 0.0;
      // (binary64 still tells the images apart below 2^30 cells)
      const double sz = Xm[2] / B[8], sy = (Xm[1] + fabs(B[5]) * sz) / B[4],
                   sx = (Xm[0] + fabs(B[1]) * sy + fabs(B[2]) * sz) / B[0];
      const double cells = fmax(sx, fmax(sy, sz));
      if (!(cells < 1e6)) slow = 1;
      if (!(cells < 4096.0)) wrap = 2;
    }
  }
  // No box: one particle far away must not cost the others their precision, nor squares
  // of bins their finite range.  From 2^16 r_max on, where float32 coordinates are a
  // 256th of r_max apart, a run's pairs are compared in binary64 and the others' grid
  // does not reach; frames within 2^17 r_max, wherever they are, need none of this.
  // One particle of N = 100,000 parked at 1e8: pair kernel 16.0 -> 4.2 ms; at 1e20, where
  // every pair was replayed and many were lost, 200.8 -> 4.2 ms.
  F.list_far = INFINITY;
  if (F.variant == V_NONE && fmax(R[0], fmax(R[1], R[2])) > 131072.0 * F.r_max) {
    F.list_far = 65536.0f * (float)F.nbins;
    far = fmin(far, 65536.0 * F.r_max);
  }
  const double side = fmax(ext[0], fmax(ext[1], ext[2]));
  for (int c = 0; c < 3; ++c) F.key_lo[c] = (float)lo[c];
  F.key_inv = side > 0.0 ? (float)(0.99999 / side) : 0.0f;
  F.wrap = wrap;
  const double cell = F.variant == V_NONE ? 0.0 : B[0] + fabs(B[1]) + fabs(B[2]) + B[4] + fabs(B[5]) + B[8];
  // positions and image vectors: the largest of them in bins; brought home, the
  // subtraction errs by 2^-52 (binary64) or 2^-45 (double-floats) of what is
  // subtracted, per axis and position
  const double reach = S * ((wrap ? ext[0] + ext[1] + ext[2] : 2.0 * far) + 2.0 * cell);
  // bins so narrow that squares of the frame's extent pass float32's range (or S itself does)
  if (!(reach < 0x1p60)) slow = 1;
  F.list_slow = slow;
  const double a0 = reach * 0x1p-44 + (wrap ? S * far * (wrap == 1 ? 0x1p-43 : 0x1p-49) : 0.0);
  // grid of the high parts: sums of positions, centres and images stay below
  // 2^23 steps, so they are exact in float32
  int e = 0;
  frexp(reach, &e);  // reach < 2^e
  F.list_grid = (float)ldexp(1.0, max(e - 22, -120));
  F.cull_abs = __double2float_ru(reach * 9.5367431640625e-07);  // 2^-20
  F.list_c0 = __double2float_ru(a0 * a0 * 0x1p28 + 0x1p-26);
  F.list_mid = __double2float_ru(4.0 * a0);
  // every decision needs the nearest integer of the root right to within one:
  // window and square-root error below a quarter bin at the far end
  const double tmax = (double)F.nbins + 40.0;
  F.list_all = !(8.0 * u * tmax + 4.0 * a0 < 0.25) || !(tmax * 4.76837158203125e-07 < 0.25);
  F.in_range = inside_one_sweep(F, sqrt(R[0] * R[0] + R[1] * R[1] + R[2] * R[2]));
}

// Derives, for one frame, the bound of the float32 decision and of the
// double-float tier from its box, r_max, nbins and the coordinate ranges found
// by stage_kernel.  Every float32 operation rounds to nearest (relative error
// <= u = 2^-24); S = nbins/r_max, t = S r, q = t^2, R_c = coordinate range.
//  t-space bound |t' - t| <= alpha*t + beta for t' = sqrt(q32) (the exact root
//  of the computed q):
//   alpha: rounding of d (none) or of the final wrapped d' (u), the
//          r^2 = fma(dz,dz,fma(dy,dy,dx*dx)) chain (3u on r^2 -> 1.5u),
//          float32 S^2 and the product q = r^2 S^2 ((eps_S2 + u)/2);
//   beta:  S*|a|, a_c the absolute error of d'_c: rounding of xj - xi (half an
//          ulp of the largest |d_c| <= R_c), of each wrap intermediate (half an
//          ulp of its largest magnitude) and the float32 box entries
//          (|k| |B32 - B|, |k| at most the nearest integer of the largest
//          |d|/L); for orthorhombic boxes, where float32 and binary64 may round
//          d/L to different images within eta of a half integer (both images
//          then have |d'_c| within eta L of L_c/2), S*2 eta L for as many
//          components as can reach L_c/2 below r_max (1 + 2/nbins).
//  q-space test: with n the integer nearest to sqrt(q32), floor(t) is decided
//  when |q32 - n^2| > (alpha t' + beta)(2 t' + 1) = 2 alpha q + (alpha + 2 beta) t' + beta;
//  load_fast_params turns it into one FMA in q (t' <= (q/tau + tau)/2 for any
//  tau > 0).
//  Tiles with a uniform image (tile_image) take beta_u: the same with their
//  own absolute errors (the image subtracted exactly, orthorhombic; the i's
//  moved by a rounded B k, triclinic).
//  double-float tier: |r2_df - r2_64| <= 2^-38 r2 + 2 r |a_mid| with |a_mid|
//  from 2^-40 times the wrap magnitudes (binary64 oracle rounding and the
//  float pair arithmetic, both far below it).
// beta also carries 2^-28 for the binary64 rounding of t itself (< 2^-29 for t < 2^22).
// If a precondition of the float32 path fails (nearest-integer range,
// triclinic margin) or the t-space bound reaches 1/4, every pair is deferred.
__device__ void window_setup(FrameDev& F, const double* R, const double* Xm) {
  const double u = 1.0 / 16777216.0;
  // binary64 input: the float32 path starts from coordinates rounded to float32,
  // each within half an ulp of the largest magnitude on its axis
  double conv[3] = {0, 0, 0};
  if (F.X64)
    for (int c = 0; c < 3; ++c) conv[c] = 2.0 * half_ulp_below(Xm[c]);
  double S = (double)F.nbins / F.r_max;
  double alpha = 3.0 * u + 0.5 * F.eps_S2;
  double a[3] = {0, 0, 0};
  double I[3] = {R[0], R[1], R[2]};  // magnitudes of the wrap intermediates (for the double-float tier)
  double tie = 0.0, tie_eps = 0.0;
  double au[3] = {0, 0, 0};  // absolute error of d'_c in tiles with a uniform image
  double aw[3][3] = {};      // the same, axis a wrapped per pair (M_AXIS + a); tie term tie_w[a]
  double tie_w[3] = {0, 0, 0};
  for (int c = 0; c < 3; ++c) {
    F.tie_m[c] = 0.0f;
    F.tie_t[c] = 0.0f;
    F.convf[c] = __double2float_ru(conv[c]);
  }
  F.kxdb = 0.0f;
  F.tie_all = 0.0f;
  F.rr2 = 0.0f;
  int all_defer = 0;
  float eps_s = 0.0f;
  const double* B = F.B;
  double dB[9];
  for (int q = 0; q < 9; ++q) {
    dB[q] = fabs((double)F.Bf[q] - B[q]);
    F.dBf[q] = __double2float_ru(dB[q]);
  }
  if (F.variant == V_ORTHO) {
    double Lmin = INFINITY, tie_c[3];
    for (int c = 0; c < 3; ++c) {
      double L = B[4 * c];
      double K = floor(R[c] / L * (1.0 + 1e-9) + 0.5);  // largest |k| = nint(d/L) over |d| <= R_c
      a[c] = half_ulp_below(R[c]) + K * dB[4 * c] + conv[c];
      I[c] = R[c] + K * L;
      if (R[c] / L > 1048576.0) all_defer = 1;  // nearest integer via the 1.5*2^23 trick needs |d/L| < 2^22
      Lmin = fmin(Lmin, L);
      // float32 and binary64 can round d/L to different images only within eta of a
      // half integer; both images then have |d'_c| within eta L of L/2
      double eta = (half_ulp_below(R[c]) + conv[c] + R[c] * fabs((double)F.invf[c] - 1.0 / L)) / L +
                   1e-15 * (R[c] / L + 1.0);
      tie_c[c] = 2.0 * eta * L;
    }
    // components that can sit at L_c/2 while t <= nbins + 1 (r <= r_max (1 + 1/nbins))
    double rr = F.r_max * (1.0 + 2.0 / (double)F.nbins);
    int m = (int)fmin(3.0, floor(4.0 * rr * rr / (Lmin * Lmin)));
    if (m >= 1) {
      double t1 = fmax(tie_c[0], fmax(tie_c[1], tie_c[2]));
      double t3 = sqrt(tie_c[0] * tie_c[0] + tie_c[1] * tie_c[1] + tie_c[2] * tie_c[2]);
      tie = S * (m >= 3 ? t3 : (m == 2 ? fmin(t3, 1.4142135623730951 * t1) : t1)) * 1.01;
    }
    tie_eps = 2.0 * fmax(tie_c[0], fmax(tie_c[1], tie_c[2])) + 1e-12 * Lmin;
    // uniform-image tiles: the image is subtracted exactly (|k| <= 1), so d'_c
    // errs only by the float32 box entry; the tie term is not needed where the
    // tile's difference range, widened by tie_m = 4 eta L, keeps one image
    for (int c = 0; c < 3; ++c) {
      au[c] = dB[4 * c] + conv[c];
      F.tie_m[c] = tie > 0.0 ? (float)(2.0 * tie_c[c]) : 0.0f;
    }
    // one axis wrapped per pair: its own error and, alone, its tie term
    for (int w = 0; w < 3; ++w) {
      for (int c = 0; c < 3; ++c) aw[w][c] = c == w ? a[c] : au[c];
      tie_w[w] = tie > 0.0 ? S * tie_c[w] * 1.01 : 0.0;
      F.tie_t[w] = __double2float_ru(tie_w[w]);
    }
    F.tie_all = __double2float_ru(tie);
    F.rr2 = __double2float_ru(rr * rr);
  } else if (F.variant == V_TRIC) {
    // sequential wrap along c, then b, then a (Eq. 5 below half the plane spacing);
    // D are the largest magnitudes of the intermediates, K the largest |k|
    double ax = B[0], bx = B[1], cx = B[2], by = B[4], cy = B[5], cz = B[8];
    double Kz = floor(R[2] / cz * (1.0 + 1e-9) + 0.5);
    double D1x = R[0] + Kz * fabs(cx), D1y = R[1] + Kz * fabs(cy);
    double Ky = floor(D1y / by * (1.0 + 1e-9) + 0.5);
    double D2x = D1x + Ky * fabs(bx);
    double Kx = floor(D2x / ax * (1.0 + 1e-9) + 0.5);
    a[0] = half_ulp_below(R[0]) + half_ulp_below(D1x) + half_ulp_below(D2x) + Kz * dB[2] + Ky * dB[1] + Kx * dB[0] +
           conv[0];
    a[1] = half_ulp_below(R[1]) + half_ulp_below(D1y) + Kz * dB[5] + Ky * dB[4] + conv[1];
    a[2] = half_ulp_below(R[2]) + Kz * dB[8] + conv[2];
    // tile images (|k| <= 1): the i's move by B k, rounded to float32 from
    // binary64 (half an ulp of the row sum), then added (half an ulp of the
    // largest |x + B k|); d = xj - x'i itself rounds relative to |d| (alpha)
    const double Sx = ax + fabs(bx) + fabs(cx), Sy = by + fabs(cy), Sz = cz;
    au[0] = half_ulp_below(Xm[0] + Sx) + half_ulp_below(Sx) + conv[0];
    au[1] = half_ulp_below(Xm[1] + Sy) + half_ulp_below(Sy) + conv[1];
    au[2] = half_ulp_below(Xm[2] + Sz) + half_ulp_below(Sz) + conv[2];
    // x wrapped per pair after the uniform c and b images (M_AXIS): d_x before
    // its wrap rounds at up to R_x + |bx| + |cx|, and the wrap adds |kx| |ax32 - ax|
    const double Dxw = R[0] + fabs(bx) + fabs(cx);
    aw[0][0] = au[0] + half_ulp_below(Dxw) + Kx * dB[0];
    aw[0][1] = au[1];
    aw[0][2] = au[2];
    F.kxdb = __double2float_ru(Kx * dB[0]);
    I[0] = D2x + Kx * ax;
    I[1] = D1y + Ky * by;
    I[2] = R[2] + Kz * cz;
    // the three nearest-integer decisions must be exact for every pair closer
    // than r_max: their float32 errors must stay below a quarter of the margin
    double ez = (2.0 * u * R[2] + conv[2] + R[2] * fabs((double)F.invf[2] * cz - 1.0)) / cz;
    double ey = (2.0 * (fmax(a[1], au[1]) + u * D1y) + D1y * fabs((double)F.invf[1] * by - 1.0)) / by;
    double ex = (2.0 * (fmax(a[0], au[0]) + u * D2x) + D2x * fabs((double)F.invf[0] * ax - 1.0)) / ax;
    double exw = (2.0 * (aw[0][0] + u * Dxw) + Dxw * fabs((double)F.invf[0] * ax - 1.0)) / ax;
    double emax = fmax(fmax(ex, exw), fmax(ey, ez));
    if (!(emax < 0.25 * (double)F.margin) || D2x / ax > 1048576.0 || D1y / by > 1048576.0 ||
        R[2] / cz > 1048576.0)
      all_defer = 1;
  } else if (F.variant == V_TRIC_SEARCH) {
    double ax = B[0], bx = B[1], cx = B[2], by = B[4], cy = B[5], cz = B[8];
    double Sz = R[2] / cz + 1.0;
    double Sy = (R[1] + fabs(cy) * Sz) / by + 1.0;
    double Sx = (R[0] + fabs(bx) * Sy + fabs(cx) * Sz) / ax + 1.0;
    double ez = 3.0 * u * (R[2] / cz + Sz);
    double ey = (3.0 * u * (R[1] + fabs(cy) * Sz) + fabs(cy) * ez) / by + 2.0 * u * Sy;
    double ex = (3.0 * u * (R[0] + fabs(bx) * Sy + fabs(cx) * Sz) + fabs(bx) * ey + fabs(cx) * ez) / ax +
                2.0 * u * Sx;
    // binary64 input: the converted coordinates move every fractional coordinate by
    // at most the sum of the conversion errors over the plane spacings
    eps_s = (float)(2.0 * fmax(ex, fmax(ey, ez)) + 4.0 * (conv[0] / ax + conv[1] / by + conv[2] / cz) + 1e-12);
    double Kx = floor(Sx + 0.5) + 1.0, Ky = floor(Sy + 0.5) + 1.0, Kz = floor(Sz + 0.5) + 1.0;
    double Ix = R[0] + Kx * ax + Ky * fabs(bx) + Kz * fabs(cx) + ax + fabs(bx) + fabs(cx);
    double Iy = R[1] + Ky * by + Kz * fabs(cy) + by + fabs(cy);
    double Iz = R[2] + Kz * cz + cz;
    a[0] = u * (R[0] + 7.0 * Ix) + (Kx + 1) * dB[0] + (Ky + 1) * dB[1] + (Kz + 1) * dB[2] + conv[0];
    a[1] = u * (R[1] + 6.0 * Iy) + (Ky + 1) * dB[4] + (Kz + 1) * dB[5] + conv[1];
    a[2] = u * (R[2] + 3.0 * Iz) + (Kz + 1) * dB[8] + conv[2];
    I[0] = Ix; I[1] = Iy; I[2] = Iz;
    if (Sx > 1048576.0 || Sy > 1048576.0 || Sz > 1048576.0 || eps_s > 0.05f) all_defer = 1;
  }
  if (F.variant == V_NONE)
    for (int c = 0; c < 3; ++c) a[c] = conv[c];  // d = xj - xi itself rounds relative to |d| (alpha)
  const double abs_u = sqrt(au[0] * au[0] + au[1] * au[1] + au[2] * au[2]);
  double beta = S * sqrt(a[0] * a[0] + a[1] * a[1] + a[2] * a[2]) * (1.0 + 64.0 * u) + tie + 1.0 / 268435456.0;
  double beta_u = (F.variant == V_ORTHO || F.variant == V_TRIC) ? S * abs_u * (1.0 + 64.0 * u) + 1.0 / 268435456.0
                                                                 : beta;
  double beta_w[3] = {beta, beta, beta};
  for (int w = 0; w < 3; ++w)
    if (F.variant == V_ORTHO || (F.variant == V_TRIC && w == 0))
      beta_w[w] = S * sqrt(aw[w][0] * aw[w][0] + aw[w][1] * aw[w][1] + aw[w][2] * aw[w][2]) * (1.0 + 64.0 * u) +
                  tie_w[w] + 1.0 / 268435456.0;
  alpha = alpha * (1.0 + 1.0 / 1024.0) + 1e-12;
  double delta = alpha * ((double)F.nbins + 1.0) + beta;
  const double beta_max = fmax(fmax(beta, beta_u), fmax(beta_w[0], fmax(beta_w[1], beta_w[2])));
  if (!(delta < 0.25) || !(alpha * ((double)F.nbins + 1.0) + beta_max < 0.25)) all_defer = 1;
  // the q-space test itself is formed per sweep (load_fast_params)
  double Imax = fmax(I[0], fmax(I[1], I[2]));
  double amid = 1.7320508075688772 * (R[0] + R[1] + R[2] + 4.0 * Imax) / 1099511627776.0;  // 2^-40
  if (F.X64)  // binary64 input: the split coordinates (2^-48 of the magnitude each) and d rounded in binary64
    amid += 1.7320508075688772 * 4.0 * fmax(conv[0], fmax(conv[1], conv[2])) / 16777216.0 +
            1.7320508075688772 * (R[0] + R[1] + R[2]) / 4503599627370496.0;
  F.mid2 = (float)(1.0 / 274877906944.0);                                                   // 2^-38
  F.mid1 = (float)(2.0 * amid / S * 1.01);
  F.tie_eps = (float)tie_eps;
  F.delta = (float)fmin(delta, 1.0);
  F.alpha_t = (float)alpha;
  F.beta_t = (float)beta;
  F.beta_u = (float)beta_u;
  for (int w = 0; w < 3; ++w) F.beta_w[w] = (float)beta_w[w];
  F.eps_s = eps_s;
  F.all_defer = all_defer;
  // no pair's root reaches the clamp: the largest possible distance is sqrt(sum R_c^2)
  {
    const double D = sqrt(R[0] * R[0] + R[1] * R[1] + R[2] * R[2]);
    F.in_range = !all_defer && inside_one_sweep(F, D);
    // no box: bounding tiles pays only when some tile can miss a sweep
    F.cull_ok = F.variant == V_NONE && (F.sweep_width < F.nbins || F.r_max < D);
  }
}

// Coordinate ranges and largest magnitudes per axis (zero for a frame without a finite coordinate).
__device__ __forceinline__ void frame_ranges(const FrameDev& F, double* R, double* Xm) {
  const bool any = F.n > 0 && F.cmin[0] <= F.cmax[0];
  for (int c = 0; c < 3; ++c) {
    const double lo = any ? (double)float_of_ord(F.cmin[c]) : 0.0, hi = any ? (double)float_of_ord(F.cmax[c]) : 0.0;
    R[c] = hi - lo;
    Xm[c] = fmax(fabs(lo), fabs(hi));
  }
}

// The spatial order's box of a frame without a box whose range is far beyond r_max, by
// one warp after list_setup, from the coordinates at x or x64.  A few particles far
// away would put all the others into one cell, and runs without an order have large
// bounds: windows as wide as the frame, no pairs left out (one particle of N = 100,000
// at 1e5: pair kernel 4.6 ms, ordered 3.1 ms).  So the box holds the bulk: the third
// smallest to the third largest of 32 particles, 30 % wider on each side.
__device__ __noinline__ void bulk_box(FrameDev& F, int lane, const float* x, const double* x64, int stride) {
  float lo[3], hi[3], range = 0.0f, side = 0.0f;
  for (int c = 0; c < 3; ++c) range = fmaxf(range, float_of_ord(F.cmax[c]) - float_of_ord(F.cmin[c]));
  if (!(range > 16.0f * F.rmax_f)) return;
  const int i = (int)((int64_t)lane * (F.n - 1) / 31);
  for (int c = 0; c < 3; ++c) {
    const int64_t at = (int64_t)i * stride + c;
    const float v = x64 ? __double2float_rn(x64[at]) : x[at];
    int rank = 0;
    for (int k = 0; k < 32; ++k) {
      const float o = __shfl_sync(kFull, v, k);
      rank += o < v || (o == v && k < lane);
    }
    const unsigned at_lo = __ballot_sync(kFull, rank == 2), at_hi = __ballot_sync(kFull, rank == 29);
    lo[c] = __shfl_sync(kFull, v, (__ffs(at_lo) - 1) & 31);
    hi[c] = __shfl_sync(kFull, v, (__ffs(at_hi) - 1) & 31);
    const float more = 0.3f * (hi[c] - lo[c]);
    lo[c] = fmaxf(lo[c] - more, float_of_ord(F.cmin[c]));
    hi[c] = fminf(hi[c] + more, float_of_ord(F.cmax[c]));
    side = fmaxf(side, hi[c] - lo[c]);
  }
  if (!(side > 0.0f && side < 0.5f * range)) return;
  __syncwarp();
  if (lane < 3) F.key_lo[lane] = lo[lane];
  if (lane == 0) F.key_inv = 0.99999f / side;
  __syncwarp();
}

// One block per frame: its descriptor in shared memory, where one thread's chain of
// dependent accesses costs a tenth of what it does in global memory, and of the two
// setups those that the frame needs: order (spatial order, list kernel) and the
// window of the tiled kernel, of which frames of the list kernel go without unless
// asked for (windows): 7 us for them, 24 with the window (24 with either before).
__global__ void frame_setup_kernel(FrameDev* frames, int order, int windows) {
  __shared__ __align__(16) FrameDev F;
  uint32_t* const dev = reinterpret_cast<uint32_t*>(frames + blockIdx.x);
  uint32_t* const own = reinterpret_cast<uint32_t*>(&F);
  for (int k = threadIdx.x; k < (int)(sizeof(FrameDev) / 4); k += blockDim.x) own[k] = dev[k];
  __syncthreads();
  if (threadIdx.x == 0) {
    double R[3], Xm[3];
    frame_ranges(F, R, Xm);
    if (order) list_setup(F, R, Xm);
    if (windows || !F.P4) window_setup(F, R, Xm);
  }
  for (int k = threadIdx.x; k < F.clear; k += blockDim.x) F.out[k] = 0ull;
  __syncwarp();
  if (order && threadIdx.x < 32 && F.variant == V_NONE && F.n > kRun)
    bulk_box(F, threadIdx.x, reinterpret_cast<const float*>(F.staged), nullptr, 4);
  __syncthreads();
  for (int k = threadIdx.x; k < (int)(sizeof(FrameDev) / 4); k += blockDim.x) dev[k] = own[k];
}

// ------------------------------------------------------------------ small frames: one launch

// Staging, list_setup and spatial order of one frame per cluster, for frames of
// which only the list kernel is run (the tiled kernel's window is not derived).
// A small frame's preparation is a chain of short steps, each over all of its
// particles: as kernels of their own (stage, setup, count, scan, scatter, bounds and
// two fills) they took 62 us at any size up to N = 5,000, most of it launches, first
// touches and one thread's binary64 arithmetic.  Here the steps meet at cluster
// barriers, the particles stay in registers, and the frame's descriptor is read into
// shared memory once.  Whole call, before -> now: N = 2,000 without a box 91 -> 64 us,
// N = 8,000 triclinic 159 -> 127 us, N = 32,000 orthorhombic 429 -> 411 us; larger
// frames have work for more SMs than a cluster's and keep the separate kernels.
static_assert((int64_t)kPrepBlock * 8 * kPrepCluster == kPrepMaxN, "particles per cluster");
// PER: particles per thread, at most, and half the counters of a pass; STRIPS: some
// species of some frame is ordered in strips (without, one pass straight through:
// three passes' code costs the smallest frames 5 us).
template <int PER, bool STRIPS>
__global__ void __launch_bounds__(kPrepBlock, 1)
    prep_kernel(const StageJob* __restrict__ jobs, const SortSeg* __restrict__ sorts, uint32_t* counts) {
  namespace cg = cooperative_groups;
  cg::cluster_group cluster = cg::this_cluster();
  constexpr int kPrepPer = PER, kPrepScan = 2 * PER;
  const int C = (int)cluster.num_blocks(), block = (int)cluster.block_rank();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int slot = block * kPrepBlock + tid, slots = C * kPrepBlock;
  __shared__ StageJob J;
  __shared__ __align__(16) FrameDev F;
  __shared__ float s_red[32][12];
  __shared__ float s_part[13];  // this block's minima (negated maxima), then 1 if a coordinate is not finite
  __shared__ float s_all[13];
  __shared__ uint32_t s_sum[32], s_total, s_base[kPrepCluster];
  __shared__ int s_bad;
  static_assert(sizeof(FrameDev) % 4 == 0 && sizeof(FrameDev) / 4 <= kPrepBlock, "one word per thread");
  const StageJob& job = jobs[blockIdx.x / C];
  if (tid == 0) {
    J = job;
    s_bad = 0;
  }
  FrameDev* const dev = job.fd;
  const int fwords = (int)(sizeof(FrameDev) / 4);
  if (tid < fwords) reinterpret_cast<uint32_t*>(&F)[tid] = reinterpret_cast<const uint32_t*>(dev)[tid];
  __syncthreads();
  const SortSeg* const S = sorts + J.sort0;
  const SortSeg& last = S[J.n_sort - 1];
  const int first_pass = STRIPS && J.strips ? 0 : 2;
  {
    const int64_t k0 = S[0].key0[first_pass], k1 = last.key0[2] + sort_keys(last, 2);
    for (int64_t k = k0 + slot; k < k1; k += slots) counts[k] = 0u;
  }
  for (int64_t k = slot; k < J.clear; k += slots) F.out[k] = 0ull;

  // ---- coordinates and their ranges
  const int n = (int)J.n, stride = J.stride;
  const double* const src64 = J.dst64 ? reinterpret_cast<const double*>(J.src) : nullptr;
  const bool frac = F.variant == V_TRIC || F.variant == V_TRIC_SEARCH;
  float3 p[kPrepPer];
  float v[12];
#pragma unroll
  for (int c = 0; c < 12; ++c) v[c] = INFINITY;
  bool bad = false;
#pragma unroll
  for (int q = 0; q < kPrepPer; ++q) {
    const int i = slot + q * slots;
    p[q] = make_float3(0.0f, 0.0f, 0.0f);
    if (i >= n) continue;
    if (src64) {
      const double* x = src64 + (int64_t)i * stride;
      p[q] = make_float3(__double2float_rn(x[0]), __double2float_rn(x[1]), __double2float_rn(x[2]));
    } else {
      const float* x = J.src + (int64_t)i * stride;
      p[q] = make_float3(x[0], x[1], x[2]);
    }
    const float3 a = p[q];
    bad |= !(isfinite(a.x) && isfinite(a.y) && isfinite(a.z));
    v[0] = fminf(v[0], a.x); v[1] = fminf(v[1], a.y); v[2] = fminf(v[2], a.z);
    v[3] = fminf(v[3], -a.x); v[4] = fminf(v[4], -a.y); v[5] = fminf(v[5], -a.z);
    if (frac) {
      const float3 s = frac_coords(F, a.x, a.y, a.z);
      v[6] = fminf(v[6], s.x); v[7] = fminf(v[7], s.y); v[8] = fminf(v[8], s.z);
      v[9] = fminf(v[9], -s.x); v[10] = fminf(v[10], -s.y); v[11] = fminf(v[11], -s.z);
    }
  }
#pragma unroll
  for (int c = 0; c < 12; ++c) {
    if (c >= 6 && !frac) break;
    for (int o = 16; o > 0; o >>= 1) v[c] = fminf(v[c], __shfl_xor_sync(kFull, v[c], o));
    if (lane == 0) s_red[warp][c] = v[c];
  }
  if (bad) s_bad = 1;
  __syncthreads();
  if (warp < 12) {
    float m = INFINITY;
    if (warp < 6 || frac) m = s_red[lane][warp];
    for (int o = 16; o > 0; o >>= 1) m = fminf(m, __shfl_xor_sync(kFull, m, o));
    if (lane == 0) s_part[warp] = m;
  }
  if (tid == 0) s_part[12] = s_bad ? -1.0f : 0.0f;
  cluster.sync();
  if (tid < 13) {
    float m = INFINITY;
    for (int b = 0; b < C; ++b) m = fminf(m, cluster.map_shared_rank(s_part, b)[tid]);
    s_all[tid] = m;
  }
  __syncthreads();

  // ---- the frame's window and grid, by every block for itself
  if (tid == 0) {
    double R[3], Xm[3];
    for (int c = 0; c < 3; ++c) {
      const float lo = s_all[c], hi = -s_all[3 + c];
      // (a frame without one finite coordinate keeps the initial, empty range)
      if (lo < INFINITY) F.cmin[c] = ord_of(lo);
      if (hi > -INFINITY) F.cmax[c] = ord_of(hi);
      if (frac && s_all[6 + c] < INFINITY) F.smin[c] = ord_of(s_all[6 + c]);
      if (frac && s_all[9 + c] < INFINITY) F.smax[c] = ord_of(-s_all[9 + c]);
    }
    F.bad = s_all[12] < 0.0f;
    frame_ranges(F, R, Xm);
    list_setup(F, R, Xm);
  }
  __syncwarp();
  if (warp == 0 && F.variant == V_NONE && n > kRun) bulk_box(F, lane, J.src, src64, stride);
  __syncthreads();
  if (block == 0 && tid < fwords) reinterpret_cast<uint32_t*>(dev)[tid] = reinterpret_cast<const uint32_t*>(&F)[tid];

  // ---- the passes of the spatial order
  int rank[kPrepPer], spec[kPrepPer];
#pragma unroll
  for (int q = 0; q < kPrepPer; ++q) {
    int a = 0, hi = J.n_sort - 1;
    while (a < hi) {
      const int mid = (a + hi + 1) >> 1;
      if (S[mid].x0 - S[mid].f0 <= slot + q * slots) a = mid; else hi = mid - 1;
    }
    spec[q] = a;
    rank[q] = 0;
  }
#pragma unroll 1
  for (int pass = STRIPS ? first_pass : 2; pass < 3; ++pass) {
    // cells, and each particle's place in its cell
    const int64_t key0 = S[0].key0[pass];
    const int keys = (int)(last.key0[pass] + sort_keys(last, pass) - key0);
    int cell[kPrepPer], place[kPrepPer];
#pragma unroll
    for (int q = 0; q < kPrepPer; ++q) {
      cell[q] = -1;
      place[q] = 0;
      const SortSeg& T = S[spec[q]];
      if (slot + q * slots >= n || (pass < 2 && T.nb[0] == 0)) continue;
      cell[q] = (int)(T.key0[pass] - key0) + sort_cell(F, T, make_float4(p[q].x, p[q].y, p[q].z, 0.0f), pass, rank[q]);
      place[q] = (int)atomicAdd(counts + key0 + cell[q], 1u);
    }
    cluster.sync();
    // prefix sum over the cells, species after species: within the block, then of
    // the blocks' totals
    const int each = (keys + slots - 1) / slots, k0 = slot * each;
    uint32_t c[kPrepScan], sum = 0u;
#pragma unroll
    for (int q = 0; q < kPrepScan; ++q) {
      c[q] = (q < each && k0 + q < keys) ? __ldcg(counts + key0 + k0 + q) : 0u;
      sum += c[q];
    }
    uint32_t incl = sum;
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t x = __shfl_up_sync(kFull, incl, o);
      if (lane >= o) incl += x;
    }
    if (lane == 31) s_sum[warp] = incl;
    __syncthreads();
    uint32_t before = s_sum[lane];
    if (warp == 0) {
      uint32_t t = before;
      for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(kFull, t, o);
      if (lane == 0) s_total = t;
    }
    if (lane >= warp) before = 0u;
    for (int o = 16; o > 0; o >>= 1) before += __shfl_xor_sync(kFull, before, o);
    uint32_t at = before + incl - sum;
#pragma unroll
    for (int q = 0; q < kPrepScan; ++q) {
      if (q < each && k0 + q < keys) __stcg(counts + key0 + k0 + q, at);
      at += c[q];
    }
    cluster.sync();
    if (tid < C) {
      uint32_t b = 0u;
      for (int r = 0; r < tid; ++r) b += *cluster.map_shared_rank(&s_total, r);
      s_base[tid] = b;
    }
    __syncthreads();
    // ranks within the species (without strips, within the frame)
    const int per_block = each * kPrepBlock;
#pragma unroll
    for (int q = 0; q < kPrepPer; ++q) {
      if (cell[q] < 0) continue;
      rank[q] = (int)(s_base[cell[q] / per_block] + __ldcg(counts + key0 + cell[q])) + place[q];
      if (STRIPS) {
        const int t0 = (int)(S[spec[q]].key0[pass] - key0);
        rank[q] -= (int)(s_base[t0 / per_block] + __ldcg(counts + key0 + t0));
      }
    }
  }

  // ---- the ordered copies
#pragma unroll
  for (int q = 0; q < kPrepPer; ++q) {
    const int i = slot + q * slots;
    if (i >= n) continue;
    const int pos = (STRIPS ? (int)(S[spec[q]].x0 - S[spec[q]].f0) : 0) + rank[q];
    const float4 a = make_float4(p[q].x, p[q].y, p[q].z, 0.0f);
    J.dst[pos] = a;
    double4 d;
    if (src64) {
      const double* x = src64 + (int64_t)i * stride;
      J.dst64[pos] = d = make_double4(x[0], x[1], x[2], 0.0);
    }
    list_position(F, a, src64 ? &d : nullptr, F.P4[pos], F.P2[pos]);
  }
  cluster.sync();

  // ---- bounds of the runs
  const int runs = last.run0 + (last.n + kRun - 1) / kRun;
  for (int r = block * 32 + warp; r < runs; r += C * 32) {
    int a = 0, hi = J.n_sort - 1;
    while (a < hi) {
      const int mid = (a + hi + 1) >> 1;
      if (S[mid].run0 <= r) a = mid; else hi = mid - 1;
    }
    run_bounds(F, S[a], r - S[a].run0, lane);
  }
}

// ------------------------------------------------------------------ A2-A8: pair kernel

// j particles per deferral-mask group: 32 pairs per lane and group without a box
// and 16 for the periodic variants (whose larger loop bodies, one per tile mode,
// outgrow the instruction cache when doubled), whatever the i particles per
// thread (mask bit = u * RI + r); the j tile is padded to kJUMax
template <int V, int RI>
constexpr int ju_of() { return (V == V_NONE ? 32 : 16) / RI; }
constexpr int kJUMax = 32;

// Tile modes of the periodic variants (tile_image): per-pair images, one
// uniform image, or a uniform image on all axes but one (M_AXIS + a:
// orthorhombic axis a; triclinic only a = 0, x), which is wrapped per pair.
// No box: M_UNI marks a tile of an in-range frame without padding, whose
// roots need no clamp.
constexpr int M_PAIR = 0, M_UNI = 1, M_AXIS = 2;
constexpr int M_SKIP = -1;  // a tile none of whose pairs has its bin in the current sweep
constexpr bool shifted_mode(int mode) { return mode >= M_UNI; }

struct FastParams {
  float S2;
  float qb1, qb0;       // near-edge bound |n^2 - q| <= qb1 q + qb0 (set_bound)
  int32_t kb1;          // bits(kMagicRound) + lo + 1
  uint32_t width;       // hi - lo
  int32_t lo, hi;       // bins [lo, hi) of this sweep
  float b[9];
  float inv[3];
  float amb_thr;        // search variant: 0.5 - eps_s
};

// The q-space test of the sweep [P.lo, P.hi) as one FMA in q.  The bound
// 2 alpha q + gamma t' + beta (gamma = alpha + 2 beta; beta of the tile mode:
// beta_t, beta_u, beta_w[a]) with t' <= (q/tau + tau)/2, true for any tau > 0,
// becomes (2 alpha + gamma/(2 tau)) q + (gamma tau/2 + beta), exact at t' = tau;
// tau = (hi + 2)/sqrt(2) (at least lo + 1) minimises the mean window over the
// sweep for pair counts growing like t^2.  The float32 evaluation (a few
// roundings, and alpha_t, beta_t rounded) is covered by the factor 1 + 2^-10.
__device__ __forceinline__ void set_bound_beta(const FrameDev& F, FastParams& P, float beta) {
  if (F.all_defer) {
    P.qb1 = P.qb0 = 1e30f;
    return;
  }
  const float tau = fmaxf((float)(P.hi + 2) * 0.70710678f, (float)(P.lo + 1));
  const float slack = 1.0f + 1.0f / 1024.0f;
  const float g = F.alpha_t + 2.0f * beta;
  P.qb1 = (2.0f * F.alpha_t + g / (2.0f * tau)) * slack;
  P.qb0 = (0.5f * g * tau + beta) * slack;
}
__device__ __forceinline__ void set_bound(const FrameDev& F, FastParams& P, int mode) {
  set_bound_beta(F, P, mode == M_PAIR ? F.beta_t : (mode == M_UNI ? F.beta_u : F.beta_w[mode - M_AXIS]));
}

// Half an ulp of the largest float32 of magnitude at most X (X >= 0, finite):
// the rounding error of any result whose magnitude X bounds.
__device__ __forceinline__ float half_ulp_f(float X) {
  return __uint_as_float(__float_as_uint(X) & 0x7f800000u) * 0x1p-24f;
}

// Largest |k| = |nint(d/L)| over |d| <= D, with room for the float32 roundings.
__device__ __forceinline__ float k_bound(float D, float inv) {
  return floorf(__fmaf_ru(D, inv * (1.0f + 0x1p-16f), 0.5f + 0x1p-16f));
}

// beta of one tile (img = (kx, ky, kz, mode) from tile_image) from the tile's
// own magnitudes instead of the frame's largest: the terms of frame_setup_kernel
// with each coordinate range, intermediate and image bound taken over the warp
// run and the j sub-chunk (imin..jmax).  Every float32 value of the tile lies
// between the rounded extreme differences (rounding is monotone), so half an ulp
// of the larger bound covers each rounding.  Orthorhombic: uniform axes err by
// |k| |L32 - L|, wrapped axes by the rounding of d = xj - xi and |k| |L32 - L|;
// the tie term of a wrapped axis a is kept only when some pair of the tile
// could lie within r_max (1 + 2/nbins) with |d'_a| near L_a/2, judged from the
// smallest displacements on the uniform axes.  Triclinic, shifted modes:
// x'_i = fl(x_i - tshift) rounds at half an ulp of the run's largest |x'|,
// tshift errs by tserr; in M_AXIS the x difference before its wrap rounds at
// half an ulp of its largest magnitude and the wrap adds |kx| |ax32 - ax|.
// Triclinic, per-pair images: the sequential wrap's intermediates.  Each is
// bounded by the frame's counterpart, so the result never exceeds the frame's
// beta of the mode; the outer factors are the same.
template <int V>
__device__ float tile_beta(const FrameDev& F, const float* imin, const float* imax, const float* jmin,
                           const float* jmax, float4 img) {
  const int mode = (int)img.w;
  const float kk[3] = {img.x, img.y, img.z};
  float a[3], tie = 0.0f;
  if (V == V_ORTHO) {
    if (mode == M_UNI) return F.beta_u;
    float mn2 = 0.0f;  // smallest squared displacement over the uniform axes (rounded down)
    for (int c = 0; c < 3; ++c) {
      if (mode == M_PAIR || mode == M_AXIS + c) {
        const float D = fmaxf(fabsf(__fsub_rn(jmin[c], imax[c])), fabsf(__fsub_rn(jmax[c], imin[c])));
        a[c] = half_ulp_f(D) + k_bound(D, F.invf[c]) * F.dBf[4 * c] + F.convf[c];
      } else {
        a[c] = fabsf(kk[c]) * F.dBf[4 * c] + F.convf[c];
        // exact displacements lie in [jmin - imax, jmax - imin] - k L, L within dBf of L32
        const float kL = kk[c] * F.Bf[4 * c];
        const float lo = __fsub_rd(__fsub_rd(jmin[c], imax[c]), kL) - F.dBf[4 * c];
        const float hi = __fsub_ru(__fsub_ru(jmax[c], imin[c]), kL) + F.dBf[4 * c];
        const float m = (lo > 0.0f) ? lo : (hi < 0.0f ? -hi : 0.0f);
        mn2 = __fmaf_rd(m, m, mn2);
      }
    }
    if (mode == M_PAIR) {
      tie = F.tie_all;
    } else {
      const int w = mode - M_AXIS;
      const float h = __fmul_rd(0.5f * F.Bf[4 * w], 1.0f - 0x1p-10f);
      if (__fmaf_rd(h, h, mn2) <= F.rr2) tie = F.tie_t[w];
    }
  } else {
    if (mode >= M_UNI) {
      const int m = 9 * (int)(kk[0] + 1.0f) + 3 * (int)(kk[1] + 1.0f) + (int)(kk[2] + 1.0f);
      for (int c = 0; c < 3; ++c) {
        const float lo = __fsub_rn(imin[c], F.tshift[m][c]), hi = __fsub_rn(imax[c], F.tshift[m][c]);
        a[c] = half_ulp_f(fmaxf(fabsf(lo), fabsf(hi))) + F.tserr[m][c] + F.convf[c];
        if (c == 0 && mode >= M_AXIS) {
          const float D = fmaxf(fabsf(__fsub_rn(jmax[0], lo)), fabsf(__fsub_rn(jmin[0], hi)));
          a[0] += half_ulp_f(D) + F.kxdb;
        }
      }
    } else {
      float D[3];
      for (int c = 0; c < 3; ++c)
        D[c] = fmaxf(fabsf(__fsub_rn(jmin[c], imax[c])), fabsf(__fsub_rn(jmax[c], imin[c])));
      const float* b = F.Bf;
      const float Kz = k_bound(D[2], F.invf[2]);
      const float D1x = __fmaf_ru(Kz, fabsf(b[2]), D[0]), D1y = __fmaf_ru(Kz, fabsf(b[5]), D[1]);
      const float Ky = k_bound(D1y, F.invf[1]);
      const float D2x = __fmaf_ru(Ky, fabsf(b[1]), D1x);
      const float Kx = k_bound(D2x, F.invf[0]);
      a[0] = half_ulp_f(D[0]) + half_ulp_f(D1x) + half_ulp_f(D2x) + Kz * F.dBf[2] + Ky * F.dBf[1] +
             Kx * F.dBf[0] + F.convf[0];
      a[1] = half_ulp_f(D[1]) + half_ulp_f(D1y) + Kz * F.dBf[5] + Ky * F.dBf[4] + F.convf[1];
      a[2] = half_ulp_f(D[2]) + Kz * F.dBf[8] + F.convf[2];
    }
  }
  const float a2 = __fmaf_ru(a[2], a[2], __fmaf_ru(a[1], a[1], __fmul_ru(a[0], a[0])));
  return __fadd_ru(__fmul_ru(__fmul_ru(F.S, __fsqrt_ru(a2)), 1.0f + 0x1p-12f), tie) + 0x1p-28f;
}

struct ItemDesc {
  FrameDev* fd;
  int32_t valid;   // 0: no more work
  int32_t h;
  int32_t pass;
  int32_t i0, ni, j0, nj;
  int32_t masked;
  int32_t skip;    // frame has no bins in this pass
};

// float32 |d'|^2 after the minimum image of the variant (NaN in, NaN out).
template <int V>
__device__ __forceinline__ float wrap_r2(float dx, float dy, float dz, const FastParams& P, bool& amb) {
  if (V == V_ORTHO) {
    dx = __fmaf_rn(-nint_scaled(dx, P.inv[0]), P.b[0], dx);
    dy = __fmaf_rn(-nint_scaled(dy, P.inv[1]), P.b[4], dy);
    dz = __fmaf_rn(-nint_scaled(dz, P.inv[2]), P.b[8], dz);
  } else if (V == V_TRIC) {
    // sequential wrap along c, b, a: the unique image inside the box-aligned brick
    float kz = nint_scaled(dz, P.inv[2]);
    dx = __fmaf_rn(-kz, P.b[2], dx);
    dy = __fmaf_rn(-kz, P.b[5], dy);
    dz = __fmaf_rn(-kz, P.b[8], dz);
    float ky = nint_scaled(dy, P.inv[1]);
    dx = __fmaf_rn(-ky, P.b[1], dx);
    dy = __fmaf_rn(-ky, P.b[4], dy);
    float kx = nint_scaled(dx, P.inv[0]);
    dx = __fmaf_rn(-kx, P.b[0], dx);
  } else if (V == V_TRIC_SEARCH) {
    // Eq. 5 wrap via back substitution, then the 27 neighbouring shifts
    float sz = __fmul_rn(dz, P.inv[2]);
    float sy = __fmul_rn(__fmaf_rn(-P.b[5], sz, dy), P.inv[1]);
    float sx = __fmul_rn(__fmaf_rn(-P.b[2], sz, __fmaf_rn(-P.b[1], sy, dx)), P.inv[0]);
    float kx = nint_f(sx), ky = nint_f(sy), kz = nint_f(sz);
    amb = (fabsf(__fsub_rn(sx, kx)) > P.amb_thr) || (fabsf(__fsub_rn(sy, ky)) > P.amb_thr) ||
          (fabsf(__fsub_rn(sz, kz)) > P.amb_thr);
    dx = __fmaf_rn(-kz, P.b[2], __fmaf_rn(-ky, P.b[1], __fmaf_rn(-kx, P.b[0], dx)));
    dy = __fmaf_rn(-kz, P.b[5], __fmaf_rn(-ky, P.b[4], dy));
    dz = __fmaf_rn(-kz, P.b[8], dz);
    float best = INFINITY;
#pragma unroll
    for (int mx = -1; mx <= 1; ++mx) {
      float ex1 = __fmaf_rn((float)mx, P.b[0], dx);
#pragma unroll
      for (int my = -1; my <= 1; ++my) {
        float ex2 = __fmaf_rn((float)my, P.b[1], ex1);
        float ey2 = __fmaf_rn((float)my, P.b[4], dy);
#pragma unroll
        for (int mz = -1; mz <= 1; ++mz) {
          float ex = __fmaf_rn((float)mz, P.b[2], ex2);
          float ey = __fmaf_rn((float)mz, P.b[5], ey2);
          float ez = __fmaf_rn((float)mz, P.b[8], dz);
          best = min_nan(best, __fmaf_rn(ez, ez, __fmaf_rn(ey, ey, __fmul_rn(ex, ex))));
        }
      }
    }
    return best;
  }
  return __fmaf_rn(dz, dz, __fmaf_rn(dy, dy, __fmul_rn(dx, dx)));
}

// float32 |d'|^2 of two pairs after the minimum image of the variant; each
// component is rounded exactly as the scalar sequence of wrap_r2.  In the
// shifted modes the caller has already subtracted the tile's images from the
// coordinates, so d is the image vector itself, but for the one axis of an
// M_AXIS mode, wrapped here as wrap_r2 does.
template <int V, int MODE = M_PAIR>
__device__ __forceinline__ float2 wrap_r2_2(float2 dx, float2 dy, float2 dz, const FastParams& P, bool& amb_a,
                                            bool& amb_b) {
  const float2 M = bc2(kMagicRound), NM = bc2(-kMagicRound);
  if (shifted_mode(MODE) && (V == V_ORTHO || V == V_TRIC)) {
    if (MODE == M_AXIS + 0) {
      float2 kx = add2(fma2(dx, bc2(P.inv[0]), M), NM);
      dx = fma2(kx, bc2(-P.b[0]), dx);
    } else if (V == V_ORTHO && MODE == M_AXIS + 1) {
      float2 ky = add2(fma2(dy, bc2(P.inv[1]), M), NM);
      dy = fma2(ky, bc2(-P.b[4]), dy);
    } else if (V == V_ORTHO && MODE == M_AXIS + 2) {
      float2 kz = add2(fma2(dz, bc2(P.inv[2]), M), NM);
      dz = fma2(kz, bc2(-P.b[8]), dz);
    }
  } else if (V == V_ORTHO) {
    float2 kx = add2(fma2(dx, bc2(P.inv[0]), M), NM);
    float2 ky = add2(fma2(dy, bc2(P.inv[1]), M), NM);
    float2 kz = add2(fma2(dz, bc2(P.inv[2]), M), NM);
    dx = fma2(kx, bc2(-P.b[0]), dx);
    dy = fma2(ky, bc2(-P.b[4]), dy);
    dz = fma2(kz, bc2(-P.b[8]), dz);
  } else if (V == V_TRIC) {
    float2 kz = add2(fma2(dz, bc2(P.inv[2]), M), NM);
    dx = fma2(kz, bc2(-P.b[2]), dx);
    dy = fma2(kz, bc2(-P.b[5]), dy);
    dz = fma2(kz, bc2(-P.b[8]), dz);
    float2 ky = add2(fma2(dy, bc2(P.inv[1]), M), NM);
    dx = fma2(ky, bc2(-P.b[1]), dx);
    dy = fma2(ky, bc2(-P.b[4]), dy);
    float2 kx = add2(fma2(dx, bc2(P.inv[0]), M), NM);
    dx = fma2(kx, bc2(-P.b[0]), dx);
  } else if (V == V_TRIC_SEARCH) {
    return make_float2(wrap_r2<V>(dx.x, dy.x, dz.x, P, amb_a), wrap_r2<V>(dx.y, dy.y, dz.y, P, amb_b));
  }
  return fma2(dz, dz, fma2(dy, dy, mul2(dx, dx)));
}

// The same with the increments of the warp aggregated in software (the hybrid
// strategy of Sec. 2.4 taken to the warp: lanes that hit one word add their
// count once): the lanes with equal addresses are found with match.any, and the
// lowest of them adds their number.  Called by all 32 lanes together.  The
// address is formed in the same instructions as count_or_defer.
__device__ __forceinline__ void count_or_defer_agg(float sm, float e, float bound, uint32_t hbase, uint32_t bit,
                                                   uint32_t& dmask) {
  asm volatile(
      "{\n\t.reg .pred pn, pl;\n\t.reg .u32 eb, sg, v, addr, peers, lm, cnt;\n\t.reg .f32 ae;\n\t"
      "mov.b32 eb, %2;\n\t"
      "shr.u32 sg, eb, 31;\n\t"
      "add.u32 v, %1, sg;\n\t"
      "shl.b32 addr, v, 2;\n\t"
      "add.u32 addr, addr, %4;\n\t"
      "abs.f32 ae, %2;\n\t"
      "setp.gtu.f32 pn, ae, %3;\n\t"
      "@!pn or.b32 %0, %0, %5;\n\t"
      "match.any.sync.b32 peers, addr, 0xffffffff;\n\t"
      "mov.u32 lm, %%lanemask_lt;\n\t"
      "and.b32 lm, lm, peers;\n\t"
      "setp.eq.u32 pl, lm, 0;\n\t"
      "popc.b32 cnt, peers;\n\t"
      "@pl red.shared.add.u32 [addr], cnt;\n\t"
      "}"
      : "+r"(dmask)
      : "r"(__float_as_uint(sm)), "f"(e), "f"(bound), "r"(hbase), "r"(bit)
      : "memory");
}

// The float32 decision of two pairs (j, j+1 against one i).  With q = r^2 S^2
// (= t^2) and n the integer nearest to the clamped root s_c, the residual
// e = n^2 - q is rounded once (fma), so its sign gives floor(t) = n or n-1, and
// |e| is compared with the bound derived in frame_setup_kernel; within it the
// pair is deferred.  The clamp (chi = hi + 1 + lane, and clo = lo - lane for
// sweeps that start above bin 0) sends far pairs to guard words with a large
// |e|, so they are not deferred; NaN pairs are never deferred.
// decide_arith2 returns sm = s_c + 1.5*2^23, e and the bound as float pairs
// (search variant: ambiguous images force the bound to +inf so the pair is
// deferred); count_or_defer acts on them.
template <int V, bool MULTI, int MODE = M_PAIR>
__device__ __forceinline__ void decide_arith2(float2 dx, float2 dy, float2 dz, const FastParams& P, float chi,
                                              float clo, float2& sm, float2& e, float2& bound) {
  bool amb_a = false, amb_b = false;
  float2 r2 = wrap_r2_2<V, MODE>(dx, dy, dz, P, amb_a, amb_b);
  float2 nq = mul2(r2, bc2(-P.S2));  // -q
  float2 sq = make_float2(sqrt_approx(-nq.x), sqrt_approx(-nq.y));
  // NaN -> chi; a no-box tile of an in-range frame (M_UNI) has neither NaN nor
  // roots near the clamp
  float2 sc = (V == V_NONE && MODE == M_UNI) ? sq : make_float2(fminf(sq.x, chi), fminf(sq.y, chi));
  if (MULTI) sc = make_float2(fmaxf(sc.x, clo), fmaxf(sc.y, clo));
  sm = add2(sc, bc2(kMagicRound));
  float2 n = add2(sm, bc2(-kMagicRound));
  e = fma2(n, n, nq);  // n^2 - q
  bound = fma2(nq, bc2(-P.qb1), bc2(P.qb0));
  if (V == V_TRIC_SEARCH) {
    if (amb_a) bound.x = INFINITY;
    if (amb_b) bound.y = INFINITY;
  }
}

// The same decision as count_or_defer, as values (used by the self check;
// single sweep, lane 0's clamp).
template <int V>
__device__ __forceinline__ void fast_decide2(float2 dx, float2 dy, float2 dz, const FastParams& P, bool& near_a,
                                             bool& near_b, uint32_t& rel_a, uint32_t& rel_b) {
  float2 sm, e, bound;
  decide_arith2<V, false>(dx, dy, dz, P, (float)(P.hi + 1), 0.0f, sm, e, bound);
  near_a = fabsf(e.x) <= bound.x;
  near_b = fabsf(e.y) <= bound.y;
  rel_a = __float_as_uint(sm.x) + (__float_as_uint(e.x) >> 31) - (uint32_t)P.kb1;
  rel_b = __float_as_uint(sm.y) + (__float_as_uint(e.y) >> 31) - (uint32_t)P.kb1;
}

// The relative bin at which the float32 path counted a pair (provisionally,
// if it deferred it): the scalar replay of decide_arith2 and count_or_defer,
// operation for operation, for the lane `src_lane` that evaluated the pair.
template <int V, bool MULTI, int MODE = M_PAIR>
__device__ __forceinline__ int provisional_rel(const FastParams& P, float4 pi, float4 pj, int src_lane,
                                               float3 ti = make_float3(0.f, 0.f, 0.f),
                                               float3 sj = make_float3(0.f, 0.f, 0.f)) {
  bool amb = false;
  float r2;
  if ((V == V_ORTHO || V == V_TRIC) && shifted_mode(MODE)) {  // the coordinates shifted by the tile's images
    float dx = __fsub_rn(__fsub_rn(pj.x, sj.x), __fsub_rn(pi.x, ti.x));
    float dy = __fsub_rn(__fsub_rn(pj.y, sj.y), __fsub_rn(pi.y, ti.y));
    float dz = __fsub_rn(__fsub_rn(pj.z, sj.z), __fsub_rn(pi.z, ti.z));
    if (MODE == M_AXIS + 0) dx = __fmaf_rn(-nint_scaled(dx, P.inv[0]), P.b[0], dx);
    if (V == V_ORTHO && MODE == M_AXIS + 1) dy = __fmaf_rn(-nint_scaled(dy, P.inv[1]), P.b[4], dy);
    if (V == V_ORTHO && MODE == M_AXIS + 2) dz = __fmaf_rn(-nint_scaled(dz, P.inv[2]), P.b[8], dz);
    r2 = __fmaf_rn(dz, dz, __fmaf_rn(dy, dy, __fmul_rn(dx, dx)));
  } else {
    r2 = wrap_r2<V>(__fadd_rn(pj.x, -pi.x), __fadd_rn(pj.y, -pi.y), __fadd_rn(pj.z, -pi.z), P, amb);
  }
  float nq = __fmul_rn(r2, -P.S2);
  float sc = fminf(sqrt_approx(-nq), (float)(P.hi + 1 + src_lane));
  if (MULTI) sc = fmaxf(sc, (float)(P.lo - src_lane));
  float sm = __fadd_rn(sc, kMagicRound);
  float n = __fadd_rn(sm, -kMagicRound);
  float e = __fmaf_rn(n, n, nq);
  return (int)(__float_as_uint(sm) + (__float_as_uint(e) >> 31) - (uint32_t)P.kb1);
}

// Bin of a deferred pair from r^2 evaluated in double-float arithmetic (about
// 44 bits, with the exact coordinate differences (float32 input; binary64
// input to about 2^-47 of the coordinate magnitude) and the same nearest images
// as the float32 path), compared with the split binary64 threshold of the
// nearest edge.  Returns -1 when even this is too close to call.  i, j:
// frame-local indices; pi, pj: the float32 coordinates.
template <int V>
__device__ int mid_bin(const FrameDev& F, int i, int j, float4 pi, float4 pj) {
  if (V == V_TRIC_SEARCH) return -1;
  DF dx, dy, dz;
  if (F.X64) {
    const double4 a = F.X64[i], b = F.X64[j];
    dx = df_diff64(b.x, a.x);
    dy = df_diff64(b.y, a.y);
    dz = df_diff64(b.z, a.z);
  } else {
    dx = two_sum(pj.x, -pi.x);
    dy = two_sum(pj.y, -pi.y);
    dz = two_sum(pj.z, -pi.z);
  }
  if (V == V_ORTHO) {
    float kx = nint_scaled(dx.h, F.invf[0]), ky = nint_scaled(dy.h, F.invf[1]), kz = nint_scaled(dz.h, F.invf[2]);
    dx = df_sub_kb(dx, kx, F.Bf[0], F.Bl[0]);
    dy = df_sub_kb(dy, ky, F.Bf[4], F.Bl[4]);
    dz = df_sub_kb(dz, kz, F.Bf[8], F.Bl[8]);
    // float32 and binary64 may pick different images near |d'_c| = L_c/2; and the
    // images must be nearest at all (the nearest integer via 1.5 2^23 is exact
    // only below 2^22 cells): the wrapped components strictly inside L_c/2
    if (fabsf(fabsf(dx.h) - 0.5f * F.Bf[0]) <= F.tie_eps || fabsf(fabsf(dy.h) - 0.5f * F.Bf[4]) <= F.tie_eps ||
        fabsf(fabsf(dz.h) - 0.5f * F.Bf[8]) <= F.tie_eps)
      return -1;
    const float lim = 0.5f - 0x1p-20f;
    if (!(fabsf(dx.h * F.invf[0]) < lim && fabsf(dy.h * F.invf[1]) < lim && fabsf(dz.h * F.invf[2]) < lim)) return -1;
  } else if (V == V_TRIC) {
    // the nearest-image integers of the float32 path, replayed exactly
    float kz = nint_scaled(dz.h, F.invf[2]);
    float fx1 = __fmaf_rn(-kz, F.Bf[2], dx.h);
    float fy1 = __fmaf_rn(-kz, F.Bf[5], dy.h);
    float ky = nint_scaled(fy1, F.invf[1]);
    float fx2 = __fmaf_rn(-ky, F.Bf[1], fx1);
    float kx = nint_scaled(fx2, F.invf[0]);
    dx = df_sub_kb(df_sub_kb(df_sub_kb(dx, kz, F.Bf[2], F.Bl[2]), ky, F.Bf[1], F.Bl[1]), kx, F.Bf[0], F.Bl[0]);
    dy = df_sub_kb(df_sub_kb(dy, kz, F.Bf[5], F.Bl[5]), ky, F.Bf[4], F.Bl[4]);
    dz = df_sub_kb(dz, kz, F.Bf[8], F.Bl[8]);
    // The images are the float32 path's; they are the exact sequential nearest
    // planes along c, b, a (Babai's step, whose vector is the minimum image of
    // every pair closer than half the smallest plane spacing) when the wrapped
    // components lie strictly inside half the periods cz, by, ax: checked here on
    // the accurate values (the frame's float32 errors may be too large for the
    // images of its float32 path, e.g. far-unwrapped coordinates).  Otherwise the
    // binary64 replay decides.
    const float lim = 0.5f - 0x1p-20f;
    if (!(fabsf(dz.h * F.invf[2]) < lim && fabsf(dy.h * F.invf[1]) < lim && fabsf(dx.h * F.invf[0]) < lim))
      return -1;
  }
  DF r2 = df_norm2(dx, dy, dz);
  float s = sqrt_approx(__fmul_rn(r2.h, F.S2));
  float n = nint_f(s);
  if (!(n >= 0.5f)) return 0;  // t below 1/2: bin 0
  if (n > (float)F.nbins) return F.nbins;
  int ni = (int)n;
  float2 T = __ldg(F.Tf + ni);
  float diff = __fadd_rn(__fsub_rn(r2.h, T.x), __fsub_rn(r2.l, T.y));
  float bound = __fmaf_rn(F.mid2, r2.h, __fmul_rn(F.mid1, s));
  if (!(fabsf(diff) > bound)) return -1;
  return diff >= 0.0f ? ni : ni - 1;
}

// The binary64 replay of one pair (about one deferred pair in 10^4): out of
// line, so that its code and registers stay out of the pair loop.
template <int V>
__device__ __noinline__ int exact_bin(const FrameDev& F, int i, int j) {
  return bin_from_thresholds(F.T, F.S, F.nbins, exact_r2<V>(F, coords64(F, i), coords64(F, j)));
}

// Exact bin of one deferred pair (frame-local indices i, j; float32 copies pi,
// pj): the double-float tier, then the binary64 replay.
template <int V>
__device__ __forceinline__ int deferred_bin(const FrameDev& F, int i, int j, float4 pi, float4 pj,
                                            unsigned& nexact) {
  int k = mid_bin<V>(F, i, j, pi, pj);
  if (k < 0) {
    k = exact_bin<V>(F, i, j);
    ++nexact;
  }
  return k;
}
// The no-box variant's drain is faster with the double-float tier out of line too.
template <int V>
__device__ __noinline__ int deferred_bin_call(const FrameDev& F, int i, int j, float4 pi, float4 pj,
                                              unsigned& nexact) {
  return deferred_bin<V>(F, i, j, pi, pj, nexact);
}

__device__ void load_fast_params(const FrameDev& F, int pass, FastParams& P);

// Decide the first `count` (<= 32) queued pairs, one per lane, move the
// provisional count of each to its exact bin where they differ, and shift the
// rest of the queue down.  A queue entry is (i - i0) | (j - j0) << 16 for the
// tile's first i and j; lane (i - i0) mod 32 evaluated the pair.
template <int V, bool MULTI, int MODE = M_PAIR>
__device__ __forceinline__ int drain_queue_body(const FrameDev* F, int pass, int i0, int j0, uint32_t* q, int qcount,
                                                uint32_t* sh, int lane, float3 ti = make_float3(0.f, 0.f, 0.f),
                                                float3 sj = make_float3(0.f, 0.f, 0.f)) {
  const int count = qcount < 32 ? qcount : 32;
  unsigned nexact = 0;
  if (lane < count) {
    const uint32_t e = q[lane];
    const int il = (int)(e & 0xFFFFu), jl = (int)(e >> 16);
    float4 pi = __ldg(F->X + i0 + il);
    float4 pj = __ldg(F->X + j0 + jl);
    FastParams P;
    load_fast_params(*F, pass, P);
    int relp = provisional_rel<V, MULTI, MODE>(P, pi, pj, il & 31, ti, sj);
    int relx = (V == V_NONE ? deferred_bin_call<V>(*F, i0 + il, j0 + jl, pi, pj, nexact)
                            : deferred_bin<V>(*F, i0 + il, j0 + jl, pi, pj, nexact)) - P.lo;
    if (relx != relp) {
      atomicAdd(sh + relp, 0xFFFFFFFFu);  // relp lies in the histogram or its guard words
      if ((uint32_t)relx < P.width) atomicAdd(sh + relx, 1u);
    }
  }
  __syncwarp();
  int rest = qcount - count;
  if (lane < rest) q[lane] = q[32 + lane];
  __syncwarp();
  for (int o = 16; o > 0; o >>= 1) nexact += __shfl_xor_sync(kFull, nexact, o);
  if (lane == 0 && nexact) atomicAdd(&const_cast<FrameDev*>(F)->exact, (unsigned long long)nexact);
  return rest;
}

template <int V, bool MULTI, int MODE = M_PAIR>
__device__ __noinline__ int drain_queue_call(const FrameDev* F, int pass, int i0, int j0, uint32_t* q, int qcount,
                                             uint32_t* sh, int lane, float3 ti = make_float3(0.f, 0.f, 0.f),
                                             float3 sj = make_float3(0.f, 0.f, 0.f)) {
  return drain_queue_body<V, MULTI, MODE>(F, pass, i0, j0, q, qcount, sh, lane, ti, sj);
}

// The register allocation of the hot loop and the size of its code decide which
// form is faster (measured): the triclinic variant keeps fewer live values across
// an inlined drain than across a call; the no-box variant is faster with the
// call, and so is the orthorhombic one, whose seven pair-loop instances (one per
// tile mode) otherwise outgrow the instruction cache (one out-of-line copy per
// mode: +0.4 % on the headline frame, +4 % on C2).
template <int V, bool MULTI, int MODE>
__device__ __forceinline__ int drain_queue(const FrameDev* F, int pass, int i0, int j0, uint32_t* q, int qcount,
                                           uint32_t* sh, int lane, float3 ti, float3 sj) {
  if constexpr (V == V_TRIC)
    return drain_queue_body<V, MULTI, MODE>(F, pass, i0, j0, q, qcount, sh, lane, ti, sj);
  else if constexpr (V == V_ORTHO)
    return drain_queue_call<V, MULTI, MODE>(F, pass, i0, j0, q, qcount, sh, lane, ti, sj);
  else
    return drain_queue_call<V, MULTI>(F, pass, i0, j0, q, qcount, sh, lane);
}

// j tile in shared memory as pairs of particles: A[p] = {x_2p, x_2p+1, y_2p, y_2p+1},
// Z[p] = {z_2p, z_2p+1}, so one LDS.128 + one LDS.64 feed two j particles.
// The i run `run` of the item (32 * RI consecutive i particles, lane + 32 r of
// it in this lane) against j particles [jb, je) of the staged tile (jb a
// multiple of kSubJ).
template <int V, bool MASKED, bool MULTI, int RI, int MODE, bool AGG>
__device__ __forceinline__ void run_tile(const FrameDev* F, const FastParams& P, const ItemDesc& it,
                                         const float4* __restrict__ sjA, const float2* __restrict__ sjZ,
                                         uint32_t* sh, uint32_t* q, int run, int lane, unsigned& ndeferred,
                                         float3 kt, int jb, int je) {
  const int ib = run * (32 * RI) + lane;
  // tile images: the image is subtracted from the coordinates, ti from the i's and
  // sj from the j's.  Orthorhombic (exact, see tile_image): k = -1 takes L from
  // the i's, k = +1 from the j's.  Triclinic: the i's move by the image vector
  // B k, rounded once (|k| <= 1, so the products are exact).
  constexpr bool SH = (V == V_ORTHO || V == V_TRIC) && shifted_mode(MODE);
  float3 ti = make_float3(0.f, 0.f, 0.f), sj = make_float3(0.f, 0.f, 0.f);
  if (V == V_ORTHO && SH) {
    ti = make_float3(kt.x < 0.f ? P.b[0] : 0.f, kt.y < 0.f ? P.b[4] : 0.f, kt.z < 0.f ? P.b[8] : 0.f);
    sj = make_float3(kt.x > 0.f ? P.b[0] : 0.f, kt.y > 0.f ? P.b[4] : 0.f, kt.z > 0.f ? P.b[8] : 0.f);
  } else if (V == V_TRIC && SH) {
    const float* v = F->tshift[9 * (int)(kt.x + 1.0f) + 3 * (int)(kt.y + 1.0f) + (int)(kt.z + 1.0f)];
    ti = make_float3(v[0], v[1], v[2]);
  }
  float2 xi[RI], yi[RI], zi[RI];  // i coordinates broadcast to both halves
#pragma unroll
  for (int r = 0; r < RI; ++r) {
    int li = ib + 32 * r;
    float x = __int_as_float(0x7fffffff), y = x, z = x;
    if (li < it.ni) {
      float4 p = __ldg(F->X + it.i0 + li);
      x = p.x; y = p.y; z = p.z;
      if (SH) {
        x = __fsub_rn(x, ti.x);
        y = __fsub_rn(y, ti.y);
        z = __fsub_rn(z, ti.z);
      }
    }
    xi[r] = bc2(-x); yi[r] = bc2(-y); zi[r] = bc2(-z);  // negated: d = xj + (-xi)
  }
  const unsigned lt_mask = (1u << lane) - 1u;
  const float qnan = __int_as_float(0x7fffffff);
  // address of bin rel = 4 (rel + kb1) + hbase (mod 2^32); clamp of the root per lane
  const uint32_t hbase = (uint32_t)__cvta_generic_to_shared(sh) - 4u * (uint32_t)P.kb1;
  const float chi = (float)(P.hi + 1 + lane);
  const float clo = (float)(P.lo - lane);
  constexpr int kJU = ju_of<V, RI>();
  const int nj4 = (je + kJU - 1) & ~(kJU - 1);  // the j tile is padded with NaN particles
  int qcount = 0;
  for (int jj0 = jb; jj0 < nj4; jj0 += kJU) {
    uint32_t dmask = 0u;
    // (u, r) are compile-time constants after unrolling: they name the mask bit
#pragma unroll
    for (int u = 0; u < kJU; u += 2) {
      const float4 A = sjA[(jj0 + u) >> 1];
      float2 Z = sjZ[(jj0 + u) >> 1];
      float2 xj = make_float2(A.x, A.y), yj = make_float2(A.z, A.w);
      if (V == V_ORTHO && SH) {  // (the wrapped axis of an M_AXIS mode has no shift)
        if (MODE != M_AXIS + 0) xj = add2(xj, bc2(-sj.x));
        if (MODE != M_AXIS + 1) yj = add2(yj, bc2(-sj.y));
        if (MODE != M_AXIS + 2) Z = add2(Z, bc2(-sj.z));
      }
#pragma unroll
      for (int r = 0; r < RI; ++r) {
        float2 dx = add2(xj, xi[r]);
        float2 dy = add2(yj, yi[r]);
        float2 dz = add2(Z, zi[r]);
        if (MASKED) {
          // intra-species: only j > i; all three components so no later test sees a number
          const int ig = it.i0 + ib + 32 * r, jg = it.j0 + jj0 + u;
          if (!(jg > ig)) { dx.x = qnan; dy.x = qnan; dz.x = qnan; }
          if (!(jg + 1 > ig)) { dx.y = qnan; dy.y = qnan; dz.y = qnan; }
        }
        float2 sm, e, bound;
        decide_arith2<V, MULTI, MODE>(dx, dy, dz, P, chi, clo, sm, e, bound);
        if (AGG) {
          count_or_defer_agg(sm.x, e.x, bound.x, hbase, 1u << (u * RI + r), dmask);
          count_or_defer_agg(sm.y, e.y, bound.y, hbase, 1u << ((u + 1) * RI + r), dmask);
        } else {
          count_or_defer(sm.x, e.x, bound.x, hbase, 1u << (u * RI + r), dmask);
          count_or_defer(sm.y, e.y, bound.y, hbase, 1u << ((u + 1) * RI + r), dmask);
        }
      }
    }
    // queue the deferred pairs: one per lane per round, compacted with a ballot
    unsigned bal = __ballot_sync(kFull, dmask != 0u);
    while (bal) {
      if (dmask) {
        int b = __ffs(dmask) - 1;
        dmask &= dmask - 1u;
        int pos = qcount + __popc(bal & lt_mask);
        q[pos] = (uint32_t)(ib + 32 * (b % RI)) | ((uint32_t)(jj0 + b / RI) << 16);
      }
      int added = __popc(bal);
      qcount += added;
      ndeferred += added;
      if (qcount >= 32) {
        __syncwarp();
        qcount = drain_queue<V, MULTI, MODE>(F, it.pass, it.i0, it.j0, q, qcount, sh, lane, ti, sj);
      }
      bal = __ballot_sync(kFull, dmask != 0u);
    }
  }
  __syncwarp();
  if (qcount > 0) drain_queue<V, MULTI, MODE>(F, it.pass, it.i0, it.j0, q, qcount, sh, lane, ti, sj);
  __syncwarp();
}

// Tiles of an item claimed dynamically: the warps take (i run, j sub-chunk)
// tiles from lists per cost class, costliest first, so that a block's warps
// reach the barrier at the end of the item within about one tile of each other
// whatever mix of tile modes and culled tiles the item holds.
constexpr int kSubPerTile = kTile / kSubJ;  // j sub-chunks per item
constexpr int kCostClasses = 3;             // per-pair images, one axis per pair, uniform image
struct TileLists {
  unsigned char* list;  // kCostClasses lists of tile indices run * kSubPerTile + c, each `cap` long
  int* count;           // per class, then the claim counter
  int cap;
};

// The cost class of a tile that runs in `mode` (after the demotion of masked tiles).
__device__ __forceinline__ int cost_class(int mode) { return mode == M_PAIR ? 0 : (mode == M_UNI ? 2 : 1); }

// The decision parameters are reloaded per item (from the L1-cached frame
// descriptor) so that only the fields of this variant are live in the loop.
// MULTI: some sweep of the launch starts above bin 0, so the root is also
// clamped from below (valid for every sweep, a separate kernel for registers).
// For the periodic variants (and no-box frames that bound their tiles) the j
// tile is taken in sub-chunks of kSubJ particles; img[t] and tbeta[t] are the
// image, mode (w) and beta of tile t = run * kSubPerTile + c, listed in `tl`.
// Masked items (the diagonal of a species block) run every tile with
// per-pair images (fewer instances).
template <int V, bool MULTI, int RI, bool AGG>
__device__ void run_item(const FrameDev* F, const ItemDesc& it, const float4* sjA, const float2* sjZ, uint32_t* sh,
                         uint32_t* q, int warp, int lane, unsigned& ndeferred, const float4* img, const float* tbeta,
                         TileLists tl, bool bounds) {
  FastParams P;
  load_fast_params(*F, it.pass, P);
  if (V == V_ORTHO || V == V_TRIC || (V == V_NONE && bounds)) {
    const int n0 = tl.count[0], n1 = n0 + tl.count[1], n = n1 + tl.count[2];
    for (;;) {
      int g = 0;
      if (lane == 0) g = atomicAdd(tl.count + kCostClasses, 1);
      g = __shfl_sync(kFull, g, 0);
      if (g >= n) break;
      const int k = g < n0 ? (int)tl.list[g] : (g < n1 ? (int)tl.list[tl.cap + g - n0] : (int)tl.list[2 * tl.cap + g - n1]);
      const int run = k / kSubPerTile, c = k - run * kSubPerTile;
      const int jb = c * kSubJ, je = min(it.nj, jb + kSubJ);
      const float3 k0 = make_float3(0.f, 0.f, 0.f);
      if (V == V_NONE) {
        if (it.masked) run_tile<V, true, MULTI, RI, M_PAIR, AGG>(F, P, it, sjA, sjZ, sh, q, run, lane, ndeferred, k0, jb, je);
        else run_tile<V, false, MULTI, RI, M_PAIR, AGG>(F, P, it, sjA, sjZ, sh, q, run, lane, ndeferred, k0, jb, je);
        continue;
      }
      const float4 im = img[k];
      const float3 kt = make_float3(im.x, im.y, im.z);
      const int mode = it.masked ? M_PAIR : (int)im.w;
      // the tile's own beta; masked tiles demoted to per-pair images take the frame's
      if (mode == (int)im.w) set_bound_beta(*F, P, tbeta[k]);
      else set_bound(*F, P, mode);
#define DH_TILE(M_, K_) run_tile<V, M_, MULTI, RI, K_, AGG>(F, P, it, sjA, sjZ, sh, q, run, lane, ndeferred, kt, jb, je)
      if (it.masked) {
        DH_TILE(true, M_PAIR);
      } else {
        switch (mode) {
          case M_UNI: DH_TILE(false, M_UNI); break;
          case M_AXIS + 0: DH_TILE(false, M_AXIS + 0); break;
          case M_AXIS + 1: if (V == V_ORTHO) DH_TILE(false, M_AXIS + 1); break;
          case M_AXIS + 2: if (V == V_ORTHO) DH_TILE(false, M_AXIS + 2); break;
          default: DH_TILE(false, M_PAIR); break;
        }
      }
#undef DH_TILE
    }
    return;
  }
  const float3 k0 = make_float3(0.f, 0.f, 0.f);
  if (it.masked) {
    run_tile<V, true, MULTI, RI, M_PAIR, AGG>(F, P, it, sjA, sjZ, sh, q, warp, lane, ndeferred, k0, 0, it.nj);
  } else if (V == V_NONE && F->in_range && it.ni == kTile && (it.nj % kJUMax) == 0) {
    // every pair real (no NaN padding) and in range: the root needs no clamp
    run_tile<V, false, MULTI, RI, M_UNI, AGG>(F, P, it, sjA, sjZ, sh, q, warp, lane, ndeferred, k0, 0, it.nj);
  } else {
    run_tile<V, false, MULTI, RI, M_PAIR, AGG>(F, P, it, sjA, sjZ, sh, q, warp, lane, ndeferred, k0, 0, it.nj);
  }
}

// The nearest-image integers of a tile pair, when the float32 per-pair path
// would compute the same ones for every pair of it.  lo/hi bound the i and j
// coordinates per axis.  The per-pair path rounds d = xj - xi, then k =
// nint(d / L) (triclinic: along c, b, a, each after the previous images are
// subtracted); every step is a correctly rounded monotone function of d, so
// the tile's extreme differences fl(jmin - imax) and fl(jmax - imin) bound the
// value of every pair at every step, and equal integers at both ends are the
// integers of every pair.  Returns (kx, ky, kz, mode): M_UNI in that case;
// M_AXIS + a when that holds for every axis but a (orthorhombic; triclinic:
// for c and b, a = 0), whose k is then 0 and wrapped per pair; M_PAIR else.
template <int V>
__device__ float4 tile_image(const FrameDev& F, const float* imin, const float* imax, const float* jmin,
                             const float* jmax) {
  float lo[3], hi[3];
  for (int c = 0; c < 3; ++c) {
    lo[c] = __fsub_rn(jmin[c], imax[c]);
    hi[c] = __fsub_rn(jmax[c], imin[c]);
  }
  const float* b = F.Bf;
  if (V == V_ORTHO) {
    // and each image must be exactly subtractable from the coordinates it moves:
    // k = +1 from the j's, k = -1 from the i's, which Sterbenz's lemma grants when
    // they lie in [L/2, 2L]
    // (widened by tie_m, so that no pair lies where float32 and binary64 may
    // round d/L to different images); an axis that fails is wrapped per pair
    float k[3];
    int nw = 0, wa = 0;
    for (int c = 0; c < 3; ++c) {
      k[c] = nint_scaled(__fsub_rn(lo[c], F.tie_m[c]), F.invf[c]);
      const float L = b[4 * c];
      bool ok = nint_scaled(__fadd_rn(hi[c], F.tie_m[c]), F.invf[c]) == k[c] &&
                ((k[c] == 0.0f) || (k[c] == 1.0f && jmin[c] >= 0.5f * L && jmax[c] <= 2.0f * L) ||
                 (k[c] == -1.0f && imin[c] >= 0.5f * L && imax[c] <= 2.0f * L));
      if (!ok) {
        ++nw;
        wa = c;
        k[c] = 0.0f;
      }
    }
    if (nw > 1) return make_float4(0.f, 0.f, 0.f, (float)M_PAIR);
    return make_float4(k[0], k[1], k[2], nw == 0 ? (float)M_UNI : (float)(M_AXIS + wa));
  } else {
    // z, then y and x after the c image, then x after the b image
    const float kz = nint_scaled(lo[2], F.invf[2]);
    if (!(nint_scaled(hi[2], F.invf[2]) == kz)) return make_float4(0.f, 0.f, 0.f, 0.f);
    float ylo = __fmaf_rn(kz, -b[5], lo[1]), yhi = __fmaf_rn(kz, -b[5], hi[1]);
    float xlo = __fmaf_rn(kz, -b[2], lo[0]), xhi = __fmaf_rn(kz, -b[2], hi[0]);
    const float ky = nint_scaled(ylo, F.invf[1]);
    if (!(nint_scaled(yhi, F.invf[1]) == ky)) return make_float4(0.f, 0.f, 0.f, 0.f);
    xlo = __fmaf_rn(ky, -b[1], xlo);
    xhi = __fmaf_rn(ky, -b[1], xhi);
    if (fabsf(ky) > 1.0f || fabsf(kz) > 1.0f) return make_float4(0.f, 0.f, 0.f, (float)M_PAIR);
    const float kx = nint_scaled(xlo, F.invf[0]);
    if (!(nint_scaled(xhi, F.invf[0]) == kx) || fabsf(kx) > 1.0f) return make_float4(0.f, ky, kz, (float)M_AXIS);
    return make_float4(kx, ky, kz, (float)M_UNI);
  }
}

// Range [lo, hi] of a real value (outward-rounded float32 bounds) and its
// distance from zero, its largest magnitude, and its distance from the lattice
// L Z for a period known to lie in [L - dL, L + dL] (all rounded so as to stay
// bounds: distances down, magnitudes up).
__device__ __forceinline__ float iv_dist0(float lo, float hi) { return lo > 0.0f ? lo : (hi < 0.0f ? -hi : 0.0f); }
__device__ __forceinline__ float iv_absmax(float lo, float hi) { return fmaxf(fabsf(lo), fabsf(hi)); }
__device__ __forceinline__ float iv_dist_lattice(float lo, float hi, float L, float dL, float invL) {
  // the nearest multiples of the period lie among m - 1 .. m + 2, m = floor(hi / L)
  // taken with the rounded reciprocal invL (within one of the exact floor)
  const float m = floorf(hi * invL);
  float d = INFINITY;
#pragma unroll
  for (int q = -1; q <= 2; ++q) {
    const float k = m + (float)q, ak = fabsf(k);
    const float x_hi = __fadd_ru(__fmul_ru(k, L), __fmul_ru(ak, dL));  // k * (true period), bounds
    const float x_lo = __fsub_rd(__fmul_rd(k, L), __fmul_ru(ak, dL));
    d = fminf(d, fmaxf(0.0f, fmaxf(__fsub_rd(lo, x_hi), __fsub_rd(x_lo, hi))));
  }
  return d;
}

// Whether no pair of a warp tile (i run bounds imin..imax, j sub-chunk bounds
// jmin..jmax, tile image img from tile_image) can have its binary64 bin in
// [lo_bin, hi_bin): then the tile contributes nothing to this sweep and is
// skipped (the tile analogue of a cell list).  Bounds on the exact minimum-image
// distance r of every pair, in float32 with directed rounding: per axis, the
// displacement range [jmin - imax, jmax - imin] (widened by the binary64-input
// conversion error), minus the tile's uniform image where it has one (the box
// vectors within their float32 rounding error dBf of binary64), or, on an axis
// wrapped per pair, at least its distance from the lattice and at most half the
// period.  Pairs with r below r_max have the same nearest images in float32 and
// binary64 (the frame's precondition), and a translate shorter than
// r_max <= h_min/2 is the minimum image, so a tile whose image-based distances all
// lie outside the sweep's distances has no pair in the sweep.  The sweep's edges
// are widened by 2^-16 (relative) for the float32 roundings here and the
// binary64 roundings of r and of floor(nbins r / r_max).  Orthorhombic: every
// mode; triclinic: uniform tiles and tiles uniform on all axes but x, and
// per-pair tiles by their z and y components alone (below).
template <int V>
__device__ bool tile_outside_sweep(const FrameDev& F, const float* imin, const float* imax, const float* jmin,
                                   const float* jmax, float4 img, int lo_bin, int hi_bin) {
  const int mode = (int)img.w;
  if (V != V_NONE && F.all_defer) return false;  // (the no-box bound needs no images)
  float lo[3], hi[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const float cv = 2.0f * F.convf[c];
    lo[c] = __fsub_rd(__fsub_rd(jmin[c], imax[c]), cv);
    hi[c] = __fadd_ru(__fsub_ru(jmax[c], imin[c]), cv);
  }
  float l[3], u[3];
  const float* b = F.Bf;
  const float* db = F.dBf;
  if (V == V_TRIC && mode == M_PAIR) {
    // Per-pair images: every image vector d - B k has z component d_z - kz cz and
    // y component d_y - ky by - kz cy, so |d - B k|^2 is at least, for its kz,
    // the z residual squared plus the distance of the y range shifted by kz cy
    // from the lattice by Z, squared.  When the z range is shorter than cz, only
    // the kz nearest to it can give less than cz^2 > r_max^2: the lower bound is
    // the minimum over those; only pairs beyond the sweep are skipped this way.
    if (!(__fsub_ru(hi[2], lo[2]) < b[8] - db[8])) return false;
    // (m is within one of the exact floor M; M - 1 .. M + 1 are the kz that matter)
    const float m = floorf(hi[2] * F.invf[2]);
    float best = INFINITY;
#pragma unroll
    for (int q = -2; q <= 2; ++q) {
      const float kz = m + (float)q, ak = fabsf(kz);
      const float sz_hi = __fadd_ru(__fmul_ru(kz, b[8]), __fmul_ru(ak, db[8]));
      const float sz_lo = __fsub_rd(__fmul_rd(kz, b[8]), __fmul_ru(ak, db[8]));
      const float sy_hi = __fadd_ru(__fmul_ru(kz, b[5]), __fmul_ru(ak, db[5]));
      const float sy_lo = __fsub_rd(__fmul_rd(kz, b[5]), __fmul_ru(ak, db[5]));
      const float dz = iv_dist0(__fsub_rd(lo[2], sz_hi), __fsub_ru(hi[2], sz_lo));
      const float dy = iv_dist_lattice(__fsub_rd(lo[1], sy_hi), __fsub_ru(hi[1], sy_lo), b[4], db[4], F.invf[1]);
      best = fminf(best, __fmaf_rd(dz, dz, __fmul_rd(dy, dy)));
    }
    const float r_hi = (hi_bin >= F.nbins) ? F.rmax_f : (float)hi_bin * F.dr_f;
    return best >= r_hi * r_hi * (1.0f + 0x1p-16f);
  }
  if (V == V_NONE) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      l[c] = iv_dist0(lo[c], hi[c]);
      u[c] = iv_absmax(lo[c], hi[c]);
    }
  } else if (V == V_ORTHO) {
    const float kk[3] = {img.x, img.y, img.z};
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const float L = b[4 * c], dL = db[4 * c];
      if (mode == M_PAIR || mode == M_AXIS + c) {  // wrapped per pair
        l[c] = iv_dist_lattice(lo[c], hi[c], L, dL, F.invf[c]);
        u[c] = __fmul_ru(__fadd_ru(L, dL), 0.5f);
      } else {  // |k| <= 1: the true shift lies in [k L32 - |k| dL, k L32 + |k| dL]
        const float s = kk[c] * L, e = fabsf(kk[c]) * dL;
        const float a = __fsub_rd(lo[c], __fadd_ru(s, e)), z = __fsub_ru(hi[c], __fsub_rd(s, e));
        l[c] = iv_dist0(a, z);
        u[c] = iv_absmax(a, z);
      }
    }
  } else {  // V_TRIC: the image vector B k (kx = 0 in the M_AXIS mode), each term |k| <= 1
    const float kx = img.x, ky = img.y, kz = img.z;
    const float ex = fabsf(kx) * db[0] + fabsf(ky) * db[1] + fabsf(kz) * db[2];
    const float ey = fabsf(ky) * db[4] + fabsf(kz) * db[5], ez = fabsf(kz) * db[8];
    const float sx_hi = __fadd_ru(__fadd_ru(__fadd_ru(kx * b[0], ky * b[1]), kz * b[2]), __fmul_ru(ex, 1.0f + 0x1p-20f));
    const float sx_lo = __fsub_rd(__fadd_rd(__fadd_rd(kx * b[0], ky * b[1]), kz * b[2]), __fmul_ru(ex, 1.0f + 0x1p-20f));
    const float sy_hi = __fadd_ru(__fadd_ru(ky * b[4], kz * b[5]), __fmul_ru(ey, 1.0f + 0x1p-20f));
    const float sy_lo = __fsub_rd(__fadd_rd(ky * b[4], kz * b[5]), __fmul_ru(ey, 1.0f + 0x1p-20f));
    const float sz_hi = __fadd_ru(kz * b[8], ez), sz_lo = __fsub_rd(kz * b[8], ez);
    const float ax = __fsub_rd(lo[0], sx_hi), bx = __fsub_ru(hi[0], sx_lo);
    const float ay = __fsub_rd(lo[1], sy_hi), by = __fsub_ru(hi[1], sy_lo);
    const float az = __fsub_rd(lo[2], sz_hi), bz = __fsub_ru(hi[2], sz_lo);
    if (mode == M_UNI) {
      l[0] = iv_dist0(ax, bx);
      u[0] = iv_absmax(ax, bx);
    } else {  // x wrapped per pair along a
      l[0] = iv_dist_lattice(ax, bx, b[0], db[0], F.invf[0]);
      u[0] = __fmul_ru(__fadd_ru(b[0], db[0]), 0.5f);
    }
    l[1] = iv_dist0(ay, by); u[1] = iv_absmax(ay, by);
    l[2] = iv_dist0(az, bz); u[2] = iv_absmax(az, bz);
  }
  const float lb2 = __fmaf_rd(l[2], l[2], __fmaf_rd(l[1], l[1], __fmul_rd(l[0], l[0])));
  const float ub2 = __fmaf_ru(u[2], u[2], __fmaf_ru(u[1], u[1], __fmul_ru(u[0], u[0])));
  // the sweep's edges in distance (squared), widened (bin width and r_max in
  // float32 from the frame descriptor: no binary64 arithmetic per tile)
  const float r_lo = (float)lo_bin * F.dr_f, r_hi = (hi_bin >= F.nbins) ? F.rmax_f : (float)hi_bin * F.dr_f;
  return (lo_bin > 0 && ub2 < r_lo * r_lo * (1.0f - 0x1p-16f)) || lb2 >= r_hi * r_hi * (1.0f + 0x1p-16f);
}

// Adds the `depth` private copies (stride words apart) bin by bin into the
// global uint64 histogram and clears them, with their guard words.
__device__ void flush_hist(uint32_t* sh, int width, int depth, int stride, uint64_t* dst, int tid) {
  const int nthreads = blockDim.x;
  for (int k = tid; k < width; k += nthreads) {
    uint32_t v = 0u;
    for (int c = 0; c < depth; ++c) {
      v += sh[c * stride + k];
      sh[c * stride + k] = 0u;
    }
    if (v) atomicAdd((unsigned long long*)(dst + k), (unsigned long long)v);
  }
  for (int k = tid; k < depth * 2 * kGuard; k += nthreads) {
    int c = k / (2 * kGuard), g = k - c * 2 * kGuard;
    sh[c * stride + (g < kGuard ? g - kGuard : width + g - kGuard)] = 0u;
  }
}

// Work item -> tile pair.  Items of a segment are numbered row by row over
// (ti, tj), i tiles of kTile particles and j tiles of kTile/jm; intra-species
// segments keep only j tiles that do not end before the i tile starts
// (tj >= jm ti), and mask pairs j <= i in those that overlap it (tj < jm (ti + 1)).
__device__ void decode_item(const PairLaunch& L, long long item, ItemDesc& it) {
  int lo = 0, hi = L.n_segs - 1;
  while (lo < hi) {
    int mid = (lo + hi + 1) >> 1;
    if (L.segs[mid].item0 <= item) lo = mid; else hi = mid - 1;
  }
  const Segment& s = L.segs[lo];
  const int jm = s.jm > 1 ? s.jm : 1;
  const int tile_j = kTile / jm;
  long long lid = item - s.item0 + s.item_base;
  int ti, tj;
  if (s.intra) {
    // row ti holds tj in [jm ti, n_tj) and starts at ti n_tj - jm ti (ti - 1) / 2
    long long n = s.n_tj;
    int a = 0, b = s.n_ti - 1;
    while (a < b) {
      int m = (a + b + 1) >> 1;
      long long start = (long long)m * n - (long long)jm * m * (m - 1) / 2;
      if (start <= lid) a = m; else b = m - 1;
    }
    ti = a;
    long long start = (long long)ti * n - (long long)jm * ti * (ti - 1) / 2;
    tj = jm * ti + (int)(lid - start);
  } else {
    ti = (int)(lid / s.n_tj);
    tj = (int)(lid - (long long)ti * s.n_tj);
  }
  it.valid = 1;
  it.fd = s.fd;
  it.h = s.h;
  it.pass = s.pass;
  it.i0 = s.a0 + ti * kTile;
  it.ni = min(kTile, s.na - ti * kTile);
  it.j0 = s.b0 + tj * tile_j;
  it.nj = min(tile_j, s.nb - tj * tile_j);
  it.masked = (s.intra && tj < jm * (ti + 1)) ? 1 : 0;
  int lo_bin = s.pass * s.fd->sweep_width;
  it.skip = (lo_bin >= s.fd->nbins) ? 1 : 0;
}

__device__ void load_fast_params(const FrameDev& F, int pass, FastParams& P) {
  int lo_bin = pass * F.sweep_width;
  int hi_bin = min(F.nbins, lo_bin + F.sweep_width);
  P.S2 = F.S2;
  P.kb1 = __float_as_int(kMagicRound) + lo_bin + 1;
  P.width = (uint32_t)(hi_bin - lo_bin);
  P.lo = lo_bin;
  P.hi = hi_bin;
#pragma unroll
  for (int c = 0; c < 9; ++c) P.b[c] = F.Bf[c];
#pragma unroll
  for (int c = 0; c < 3; ++c) P.inv[c] = F.invf[c];
  P.amb_thr = 0.5f - F.eps_s;
  set_bound(F, P, M_PAIR);
}

// One instance per minimum-image variant V (every segment of the launch has a
// frame of that variant) and per MULTI.
// Register budgets: 256-thread blocks keep three blocks per SM (80 registers)
// for the no-box and orthorhombic variants, two (128 registers: the triclinic
// loop spills at 80, which costs more than the third block gains); 512- and
// 1024-thread blocks, meant for wide histograms, one.
template <int V, int RI>
constexpr int min_blocks_per_sm() {
  return RI < 4 ? 1 : ((V == V_NONE || V == V_ORTHO) ? 3 : 2);
}

// AGG: the increments of a warp aggregated in software (count_or_defer_agg).
template <int V, bool MULTI, int RI, bool AGG = false>
__global__ void __launch_bounds__(kTile / RI, min_blocks_per_sm<V, RI>()) pair_kernel(PairLaunch L) {
  constexpr int BLOCK = kTile / RI;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  // `depth` private histogram copies, each [kGuard guard words | bins | kGuard
  // guard words] (stride words), then the j tile and the per-warp queues
  const int depth = L.hist_depth > 1 ? L.hist_depth : 1;
  const int stride = ((L.hist_width + 3) & ~3) + 2 * kGuard;
  uint32_t* hist0 = reinterpret_cast<uint32_t*>(smem_raw) + kGuard;
  float4* sjA = reinterpret_cast<float4*>(reinterpret_cast<uint32_t*>(smem_raw) + depth * stride);
  float2* sjZ = reinterpret_cast<float2*>(sjA + kTile / 2);
  uint32_t* sq = reinterpret_cast<uint32_t*>(sjZ + kTile / 2);
  __shared__ ItemDesc s_it;
  constexpr bool kTileImage = (V == V_ORTHO || V == V_TRIC);
  // tile bounds: always with tile images; without a box for frames whose tiles
  // can miss a sweep (FrameDev::cull_ok), for culling only
  constexpr bool kTileBounds = kTileImage || V == V_NONE;
  // per j sub-chunk: j min xyz, j max xyz; per warp and sub-chunk: the tile image
  __shared__ float s_bnd[kTileBounds ? kTile / kSubJ : 1][6];
  __shared__ float4 s_img[kTileBounds ? BLOCK / 32 : 1][kTileBounds ? kTile / kSubJ : 1];
  __shared__ float s_beta[kTileImage ? BLOCK / 32 : 1][kTileImage ? kTile / kSubJ : 1];  // per-tile beta
  static_assert(!kTileBounds || BLOCK / 32 >= kTile / kSubJ, "one warp per j sub-chunk");
  // the item's tiles to run, per cost class, and the counters of run_item
  constexpr int kListCap = kTileBounds ? (BLOCK / 32) * kSubPerTile : 1;
  static_assert(kListCap <= 256, "tile indices fit a byte");
  __shared__ unsigned char s_list[kTileBounds ? kCostClasses : 1][kListCap];
  __shared__ int s_cnt[kCostClasses + 1];

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  uint32_t* q = sq + warp * kQueueCap;
  uint32_t* sh = hist0 + (warp % depth) * stride;  // this warp's copy
  for (int k = tid; k < depth * stride; k += BLOCK) reinterpret_cast<uint32_t*>(smem_raw)[k] = 0u;

  const FrameDev* cur_fd = nullptr;
  int cur_h = -1, cur_pass = -1;
  unsigned long long since = 0;  // pairs accumulated in sh since the last flush
  uint64_t* cur_dst = nullptr;
  int cur_width = 0;

  // Guided self-scheduling: thread 0 claims runs of consecutive items whose
  // length shrinks with the work left (at most 64, at least 1), so a block
  // mostly stays on one segment (few histogram flushes) and the tail stays fine.
  long long run_next = 0, run_end = 0;
  for (;;) {
    if (tid == 0) {
      if (run_next >= run_end) {
        long long cur = (long long)*(volatile unsigned long long*)&L.ctl->next_item;
        long long ch = (L.n_items - cur) / (4LL * gridDim.x);
        ch = ch < 1 ? 1 : (ch > 64 ? 64 : ch);
        run_next = (long long)atomicAdd(&L.ctl->next_item, (unsigned long long)ch);
        run_end = run_next + ch < (long long)L.n_items ? run_next + ch : (long long)L.n_items;
      }
      long long item = run_next++;
      if (item >= L.n_items) s_it.valid = 0;
      else decode_item(L, item, s_it);
      for (int k = 0; k <= kCostClasses; ++k) s_cnt[k] = 0;
    }
    __syncthreads();
    const ItemDesc it = s_it;
    if (!it.valid) break;
    if (!it.skip) {
      const FrameDev& F = *it.fd;
      const unsigned long long pairs = (unsigned long long)it.ni * (unsigned long long)it.nj;
      if (it.fd != cur_fd || it.h != cur_h || it.pass != cur_pass || since + pairs > 0xFFFFFFFFull) {
        if (cur_fd) {
          __syncthreads();
          flush_hist(hist0, cur_width, depth, stride, cur_dst, tid);
          __syncthreads();
        }
        int lo_bin = it.pass * F.sweep_width;
        cur_fd = it.fd;
        cur_h = it.h;
        cur_pass = it.pass;
        cur_width = min(F.nbins, lo_bin + F.sweep_width) - lo_bin;
        cur_dst = F.out + (size_t)it.h * F.nbins + lo_bin;
        since = 0;
      }
      since += pairs;
      // stage the j tile in pair layout, padded with NaN particles to a multiple of kJUMax
      const int nj4 = (it.nj + kJUMax - 1) & ~(kJUMax - 1);
      for (int k = tid; k < nj4; k += BLOCK) {
        float4 v = k < it.nj ? __ldg(F.X + it.j0 + k)
                             : make_float4(__int_as_float(0x7fffffff), __int_as_float(0x7fffffff),
                                           __int_as_float(0x7fffffff), 0.f);
        float* a = reinterpret_cast<float*>(sjA + (k >> 1));
        a[k & 1] = v.x;
        a[2 + (k & 1)] = v.y;
        reinterpret_cast<float*>(sjZ + (k >> 1))[k & 1] = v.z;
      }
      // tile images: the bounds of this warp's i run against those of each
      // j sub-chunk of kSubJ particles (warp c reduces sub-chunk c)
      float ib_[6] = {INFINITY, INFINITY, INFINITY, -INFINITY, -INFINITY, -INFINITY};
      const bool bounds = kTileImage || (V == V_NONE && F.cull_ok);  // the same for the whole block
      if (bounds) {
        const int ib = warp * (32 * RI) + lane;  // this warp's i run (the particles run_tile gives it)
        for (int r = 0; r < RI; ++r) {
          const int li = ib + 32 * r;
          if (li < it.ni) {
            float4 v = __ldg(F.X + it.i0 + li);
            ib_[0] = fminf(ib_[0], v.x); ib_[1] = fminf(ib_[1], v.y); ib_[2] = fminf(ib_[2], v.z);
            ib_[3] = fmaxf(ib_[3], v.x); ib_[4] = fmaxf(ib_[4], v.y); ib_[5] = fmaxf(ib_[5], v.z);
          }
        }
        for (int o = 16; o > 0; o >>= 1)
          for (int a = 0; a < 6; ++a) {
            float other = __shfl_xor_sync(kFull, ib_[a], o);
            ib_[a] = a < 3 ? fminf(ib_[a], other) : fmaxf(ib_[a], other);
          }
      }
      __syncthreads();
      if (bounds) {
        if (warp * kSubJ < it.nj) {
          float jm[6] = {INFINITY, INFINITY, INFINITY, -INFINITY, -INFINITY, -INFINITY};
          const int ke = min(it.nj, (warp + 1) * kSubJ);
          for (int k = warp * kSubJ + lane; k < ke; k += 32) {
            const float* a = reinterpret_cast<const float*>(sjA + (k >> 1));
            const float x = a[k & 1], y = a[2 + (k & 1)];
            const float z = reinterpret_cast<const float*>(sjZ + (k >> 1))[k & 1];
            jm[0] = fminf(jm[0], x); jm[1] = fminf(jm[1], y); jm[2] = fminf(jm[2], z);
            jm[3] = fmaxf(jm[3], x); jm[4] = fmaxf(jm[4], y); jm[5] = fmaxf(jm[5], z);
          }
          for (int o = 16; o > 0; o >>= 1)
            for (int a = 0; a < 6; ++a) {
              float other = __shfl_xor_sync(kFull, jm[a], o);
              jm[a] = a < 3 ? fminf(jm[a], other) : fmaxf(jm[a], other);
            }
          if (lane == 0)
            for (int a = 0; a < 6; ++a) s_bnd[warp][a] = jm[a];
        }
        __syncthreads();
        const int ni_w = min(32 * RI, it.ni - warp * 32 * RI);  // i particles of this warp
        const int lo_bin = it.pass * F.sweep_width, hi_bin = min(F.nbins, lo_bin + F.sweep_width);
        for (int c = 0; c * kSubJ < it.nj; ++c) {
          float4 img = make_float4(0.f, 0.f, 0.f, 0.f);
          float tb = 0.0f;
          if (kTileImage) {
            if (ni_w > 0) img = tile_image<V>(F, ib_, ib_ + 3, s_bnd[c], s_bnd[c] + 3);
            tb = tile_beta<V>(F, ib_, ib_ + 3, s_bnd[c], s_bnd[c] + 3, img);
          }
          const unsigned long long np =
              (unsigned long long)max(ni_w, 0) * (unsigned long long)(min(it.nj, (c + 1) * kSubJ) - c * kSubJ);
          const bool skip = ni_w > 0 && tile_outside_sweep<V>(F, ib_, ib_ + 3, s_bnd[c], s_bnd[c] + 3, img, lo_bin,
                                                             hi_bin);
          if (lane == 0) {
            if (skip) {
              img.w = (float)M_SKIP;
              atomicAdd(&it.fd->culled_pairs, np);
            } else if (img.w == (float)M_UNI) {
              atomicAdd(&it.fd->uniform_pairs, np);
            } else if (img.w >= (float)M_AXIS) {
              atomicAdd(&it.fd->axis_pairs, np);
            }
            s_img[warp][c] = img;
            if (kTileImage) s_beta[warp][c] = tb;
            if (!skip && ni_w > 0) {
              const int cls = cost_class(it.masked ? M_PAIR : (int)img.w);
              s_list[cls][atomicAdd(&s_cnt[cls], 1)] = (unsigned char)(warp * kSubPerTile + c);
            }
          }
        }
        __syncthreads();  // every tile listed
      }
      unsigned ndef = 0;
      run_item<V, MULTI, RI, AGG>(it.fd, it, sjA, sjZ, sh, q, warp, lane, ndef, &s_img[0][0], &s_beta[0][0],
                                  TileLists{&s_list[0][0], s_cnt, kListCap}, bounds);
      if (lane == 0 && ndef) atomicAdd(&it.fd->deferred, (unsigned long long)ndef);
    }
    __syncthreads();
  }
  if (cur_fd) {
    __syncthreads();
    flush_hist(hist0, cur_width, depth, stride, cur_dst, tid);
  }
}

// ------------------------------------------------------------------ self checks

// Largest relative error of sqrt.approx.ftz.f32 over every float in [1, 4)
// (two binades: the relative error pattern repeats with the exponent's parity),
// against the correctly rounded binary64 square root.
__global__ void check_sqrt_kernel(unsigned long long* max_err_bits) {
  const uint32_t base = 0x3F800000u;  // 1.0f
  const uint32_t count = 2u << 23;    // [1, 4)
  double worst = 0.0;
  for (uint32_t k = blockIdx.x * blockDim.x + threadIdx.x; k < count; k += gridDim.x * blockDim.x) {
    float x = __uint_as_float(base + k);
    double ref = __dsqrt_rn((double)x);
    double e = fabs((double)sqrt_approx(x) - ref) / ref;
    worst = fmax(worst, e);
  }
  for (int o = 16; o > 0; o >>= 1) worst = fmax(worst, __shfl_xor_sync(kFull, worst, o));
  if ((threadIdx.x & 31) == 0) atomicMax(max_err_bits, (unsigned long long)__double_as_longlong(worst));
}

// splitmix64: a counter-based generator for the sampled pairs
__device__ __forceinline__ uint64_t mix64(uint64_t z) {
  z += 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

// For sampled pairs of one frame, the decision rule against the binary64
// definition: out[0] = max |sqrt(q32) - t64| / (alpha t64 + beta) over pairs
// inside the histogram (bits of a double; the analysis says < 1); out[1] =
// pairs whose float32 or double-float decision differs from the binary64 bin
// (must be 0); out[2] = pairs compared.
template <int V>
__device__ void check_window_pair(const FrameDev& F, const FastParams& P, int i, int j, double* worst,
                                  unsigned long long* viol, unsigned long long* checked) {
  float4 pi = F.X[i], pj = F.X[j];
  bool nearedge, nb_unused;
  uint32_t rel, rb_unused;
  const float2 dx = bc2(__fsub_rn(pj.x, pi.x)), dy = bc2(__fsub_rn(pj.y, pi.y)), dz = bc2(__fsub_rn(pj.z, pi.z));
  fast_decide2<V>(dx, dy, dz, P, nearedge, nb_unused, rel, rb_unused);
  bool amb0 = false, amb1 = false;
  float q = __fmul_rn(wrap_r2_2<V>(dx, dy, dz, P, amb0, amb1).x, P.S2);
  double r2 = exact_r2<V>(F, coords64(F, i), coords64(F, j));
  int k64 = bin_from_thresholds(F.T, F.S, F.nbins, r2);
  double t64 = __dmul_rn(__dsqrt_rn(r2), (double)F.nbins / F.r_max);
  if (t64 < (double)F.nbins + 1.0 && isfinite(q)) {
    double tq = __dsqrt_rn((double)q);
    *worst = fmax(*worst, fabs(tq - t64) / ((double)F.alpha_t * t64 + (double)F.beta_t));
    ++*checked;
  }
  if (!nearedge) {
    int k32 = (int)rel;  // lo = 0 here
    if (rel > (uint32_t)F.nbins) k32 = F.nbins;
    if (k32 != k64) ++*viol;
  } else {
    int km = mid_bin<V>(F, i, j, pi, pj);
    if (km >= 0 && km != k64) ++*viol;
  }
}

__global__ void check_window_kernel(const FrameDev* Fp, uint64_t n_samples, uint64_t seed,
                                    unsigned long long* out) {
  const FrameDev& F = *Fp;
  FastParams P;
  load_fast_params(F, 0, P);
  P.width = (uint32_t)F.nbins;  // decide over the whole histogram
  P.hi = F.nbins;
  double worst = 0.0;
  unsigned long long viol = 0, checked = 0;
  if (F.n >= 2) {
    for (uint64_t s = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; s < n_samples;
         s += (uint64_t)gridDim.x * blockDim.x) {
      uint64_t h = mix64(seed ^ mix64(s));
      int i = (int)(h % (uint64_t)F.n);
      int j = (int)((h >> 32) % (uint64_t)F.n);
      if (i == j) continue;
      switch (F.variant) {
        case V_NONE: check_window_pair<V_NONE>(F, P, i, j, &worst, &viol, &checked); break;
        case V_ORTHO: check_window_pair<V_ORTHO>(F, P, i, j, &worst, &viol, &checked); break;
        case V_TRIC: check_window_pair<V_TRIC>(F, P, i, j, &worst, &viol, &checked); break;
        default: check_window_pair<V_TRIC_SEARCH>(F, P, i, j, &worst, &viol, &checked); break;
      }
    }
  }
  for (int o = 16; o > 0; o >>= 1) {
    worst = fmax(worst, __shfl_xor_sync(kFull, worst, o));
    viol += __shfl_xor_sync(kFull, viol, o);
    checked += __shfl_xor_sync(kFull, checked, o);
  }
  if ((threadIdx.x & 31) == 0) {
    atomicMax(out, (unsigned long long)__double_as_longlong(worst));
    atomicAdd(out + 1, viol);
    atomicAdd(out + 2, checked);
  }
}

cudaError_t launch_check_sqrt(unsigned long long* out, cudaStream_t stream) {
  clear_stale_error();
  check_sqrt_kernel<<<1024, 256, 0, stream>>>(out);
  return cudaGetLastError();
}

cudaError_t launch_check_window(const FrameDev* F, uint64_t n_samples, uint64_t seed, unsigned long long* out,
                                cudaStream_t stream) {
  clear_stale_error();
  check_window_kernel<<<1024, 256, 0, stream>>>(F, n_samples, seed, out);
  return cudaGetLastError();
}

// The tile modes against their own bounds: one pair of a tile evaluated with the
// arithmetic of run_tile in mode MODE (coordinates shifted by the tile's images,
// then decide_arith2 with the tile's bound), against the binary64 bin.
template <int V, int MODE>
__device__ void check_tile_pair(const FrameDev& F, const FastParams& P, float beta, float3 kt, int i, int j,
                                double* worst, unsigned long long* viol, unsigned long long* checked) {
  const float4 pi = F.X[i], pj = F.X[j];
  float3 ti = make_float3(0.f, 0.f, 0.f), sj = make_float3(0.f, 0.f, 0.f);
  if (V == V_ORTHO && MODE >= M_UNI) {
    ti = make_float3(kt.x < 0.f ? P.b[0] : 0.f, kt.y < 0.f ? P.b[4] : 0.f, kt.z < 0.f ? P.b[8] : 0.f);
    sj = make_float3(kt.x > 0.f ? P.b[0] : 0.f, kt.y > 0.f ? P.b[4] : 0.f, kt.z > 0.f ? P.b[8] : 0.f);
  } else if (V == V_TRIC && MODE >= M_UNI) {
    const float* v = F.tshift[9 * (int)(kt.x + 1.0f) + 3 * (int)(kt.y + 1.0f) + (int)(kt.z + 1.0f)];
    ti = make_float3(v[0], v[1], v[2]);
  }
  const float2 dx = bc2(__fsub_rn(__fsub_rn(pj.x, sj.x), __fsub_rn(pi.x, ti.x)));
  const float2 dy = bc2(__fsub_rn(__fsub_rn(pj.y, sj.y), __fsub_rn(pi.y, ti.y)));
  const float2 dz = bc2(__fsub_rn(__fsub_rn(pj.z, sj.z), __fsub_rn(pi.z, ti.z)));
  float2 sm, e, bound;
  decide_arith2<V, false, MODE>(dx, dy, dz, P, (float)(P.hi + 1), 0.0f, sm, e, bound);
  bool amb0 = false, amb1 = false;
  const float q = __fmul_rn(wrap_r2_2<V, MODE>(dx, dy, dz, P, amb0, amb1).x, P.S2);
  const double r2 = exact_r2<V>(F, coords64(F, i), coords64(F, j));
  const int k64 = bin_from_thresholds(F.T, F.S, F.nbins, r2);
  const double t64 = __dmul_rn(__dsqrt_rn(r2), (double)F.nbins / F.r_max);
  if (t64 < (double)F.nbins + 1.0 && isfinite(q)) {
    *worst = fmax(*worst, fabs(__dsqrt_rn((double)q) - t64) / ((double)F.alpha_t * t64 + (double)beta));
    ++*checked;
  }
  if (!(fabsf(e.x) <= bound.x)) {
    const uint32_t rel = __float_as_uint(sm.x) + (__float_as_uint(e.x) >> 31) - (uint32_t)P.kb1;
    const int k32 = rel > (uint32_t)F.nbins ? F.nbins : (int)rel;
    if (k32 != k64) ++*viol;
  }
}

// One block per sampled tile: a run of 128 consecutive particles (the i's of one
// warp of a 256-thread block) and a j sub-chunk of kSubJ, at random aligned
// starts.  out[0] = largest |t32 - t64| / (alpha t64 + beta_tile) (must be < 1),
// out[1] = pairs decided in float32 with a bin other than the binary64 one (must
// be 0), out[2] = pairs compared, out[3] = sampled tiles in a shifted mode.
template <int V>
__global__ void check_tiles_kernel(const FrameDev* Fp, uint64_t n_tiles, uint64_t seed, unsigned long long* out) {
  const FrameDev& F = *Fp;
  FastParams P;
  load_fast_params(F, 0, P);
  P.width = (uint32_t)F.nbins;
  P.hi = F.nbins;
  __shared__ float s_b[8][6];
  __shared__ float s_bnd[12];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  double worst = 0.0;
  unsigned long long viol = 0, checked = 0, shifted = 0;
  const int ni = min(128, F.n), nj = min(kSubJ, F.n);
  for (uint64_t s = blockIdx.x; s < n_tiles; s += gridDim.x) {
    const uint64_t h = mix64(seed ^ mix64(s));
    const int i0 = (int)((h % (uint64_t)((F.n - ni) / 128 + 1)) * 128);
    const int j0 = (int)(((h >> 32) % (uint64_t)((F.n - nj) / kSubJ + 1)) * kSubJ);
    for (int part = 0; part < 2; ++part) {  // bounds of the i run, then of the j chunk
      const int b0 = part ? j0 : i0, nb = part ? nj : ni;
      float m[6] = {INFINITY, INFINITY, INFINITY, -INFINITY, -INFINITY, -INFINITY};
      for (int k = threadIdx.x; k < nb; k += blockDim.x) {
        const float4 v = F.X[b0 + k];
        m[0] = fminf(m[0], v.x); m[1] = fminf(m[1], v.y); m[2] = fminf(m[2], v.z);
        m[3] = fmaxf(m[3], v.x); m[4] = fmaxf(m[4], v.y); m[5] = fmaxf(m[5], v.z);
      }
      for (int o = 16; o > 0; o >>= 1)
        for (int a = 0; a < 6; ++a) {
          const float other = __shfl_xor_sync(kFull, m[a], o);
          m[a] = a < 3 ? fminf(m[a], other) : fmaxf(m[a], other);
        }
      if (lane == 0)
        for (int a = 0; a < 6; ++a) s_b[warp][a] = m[a];
      __syncthreads();
      if (threadIdx.x < 6) {
        float v = s_b[0][threadIdx.x];
        for (int w = 1; w < 8; ++w)
          v = threadIdx.x < 3 ? fminf(v, s_b[w][threadIdx.x]) : fmaxf(v, s_b[w][threadIdx.x]);
        s_bnd[6 * part + threadIdx.x] = v;
      }
      __syncthreads();
    }
    const float4 img = tile_image<V>(F, s_bnd, s_bnd + 3, s_bnd + 6, s_bnd + 9);
    const float beta = tile_beta<V>(F, s_bnd, s_bnd + 3, s_bnd + 6, s_bnd + 9, img);
    FastParams Q = P;
    set_bound_beta(F, Q, beta);
    const float3 kt = make_float3(img.x, img.y, img.z);
    if (threadIdx.x == 0 && img.w >= (float)M_UNI) ++shifted;
    for (int k = threadIdx.x; k < ni * nj; k += blockDim.x) {
      const int i = i0 + k % ni, j = j0 + k / ni;
      if (i == j) continue;
      switch ((int)img.w) {
        case M_UNI: check_tile_pair<V, M_UNI>(F, Q, beta, kt, i, j, &worst, &viol, &checked); break;
        case M_AXIS + 0: check_tile_pair<V, M_AXIS + 0>(F, Q, beta, kt, i, j, &worst, &viol, &checked); break;
        case M_AXIS + 1:
          if (V == V_ORTHO) check_tile_pair<V, M_AXIS + 1>(F, Q, beta, kt, i, j, &worst, &viol, &checked);
          break;
        case M_AXIS + 2:
          if (V == V_ORTHO) check_tile_pair<V, M_AXIS + 2>(F, Q, beta, kt, i, j, &worst, &viol, &checked);
          break;
        default: check_tile_pair<V, M_PAIR>(F, Q, beta, kt, i, j, &worst, &viol, &checked); break;
      }
    }
    __syncthreads();  // s_b, s_bnd are rewritten by the next tile
  }
  for (int o = 16; o > 0; o >>= 1) {
    worst = fmax(worst, __shfl_xor_sync(kFull, worst, o));
    viol += __shfl_xor_sync(kFull, viol, o);
    checked += __shfl_xor_sync(kFull, checked, o);
    shifted += __shfl_xor_sync(kFull, shifted, o);
  }
  if (lane == 0) {
    atomicMax(out, (unsigned long long)__double_as_longlong(worst));
    atomicAdd(out + 1, viol);
    atomicAdd(out + 2, checked);
    atomicAdd(out + 3, shifted);
  }
}

cudaError_t launch_check_tiles(const FrameDev* F, int variant, uint64_t n_tiles, uint64_t seed,
                               unsigned long long* out, cudaStream_t stream) {
  clear_stale_error();
  if (variant == V_ORTHO) check_tiles_kernel<V_ORTHO><<<456, 256, 0, stream>>>(F, n_tiles, seed, out);
  else if (variant == V_TRIC) check_tiles_kernel<V_TRIC><<<456, 256, 0, stream>>>(F, n_tiles, seed, out);
  else return cudaErrorInvalidValue;
  return cudaGetLastError();
}


// ------------------------------------------------------------------ g(r), Eq. 1

// g = (counts / n_frames) / (pair density x shell volume) per bin, binary64.
// The shell of bin k, (4 pi / 3)(r_{k+1}^3 - r_k^3) with r_k = k dr, is
// evaluated as (4 pi / 3) dr^3 (3k(k+1) + 1): the integer factor is exact for
// k < 2^25, so no cancellation between the two cubes.
__global__ void rdf_kernel(const uint64_t* __restrict__ counts, int32_t n_hist, int32_t nbins, double r_max,
                           const double* __restrict__ dens, uint64_t n_frames, double* __restrict__ g) {
  const int64_t total = (int64_t)n_hist * nbins;
  const double dr = __ddiv_rn(r_max, (double)nbins);
  const double c = __dmul_rn(__dmul_rn(4.0 * 3.14159265358979323846 / 3.0, dr), __dmul_rn(dr, dr));
  for (int64_t idx = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; idx < total;
       idx += (int64_t)gridDim.x * blockDim.x) {
    const int32_t h = (int32_t)(idx / nbins);
    const double k = (double)(idx - (int64_t)h * nbins);
    const double poly = __fma_rn(__dmul_rn(3.0, k), __dadd_rn(k, 1.0), 1.0);
    const double per_frame = __ddiv_rn((double)counts[idx], (double)n_frames);
    g[idx] = __ddiv_rn(per_frame, __dmul_rn(dens[h], __dmul_rn(c, poly)));
  }
}

cudaError_t launch_rdf(const uint64_t* counts, int32_t n_hist, int32_t nbins, double r_max,
                       const double* pair_density, uint64_t n_frames, double* g, cudaStream_t stream) {
  clear_stale_error();
  int64_t total = (int64_t)n_hist * nbins;
  int blocks = (int)std::min<int64_t>((total + 255) / 256, 4096);
  rdf_kernel<<<blocks, 256, 0, stream>>>(counts, n_hist, nbins, r_max, pair_density, n_frames, g);
  return cudaGetLastError();
}

// ------------------------------------------------------------------ launchers


size_t pair_kernel_smem(int hist_width, int depth, int block) {
  size_t stride = (size_t)((hist_width + 3) & ~3) + 2 * kGuard;
  size_t warps = (size_t)(block == kBlockHuge ? kBlockHuge : block == kBlockLarge ? kBlockLarge : kBlockSmall) / 32;
  return (size_t)(depth > 1 ? depth : 1) * stride * 4 + (size_t)kTile * 12 + warps * kQueueCap * 4;
}

int pair_kernel_max_width() {
  int dev = 0;
  cudaGetDevice(&dev);
  int optin = 0;
  cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  size_t fixed = pair_kernel_smem(0) + sizeof(ItemDesc) + 64;
  if ((size_t)optin <= fixed) return 0;
  return (int)(((size_t)optin - fixed) / 4) & ~3;
}

// Blocks of both instances that fit on one SM with `smem` bytes of dynamic
// shared memory; 0 (and no error left behind) when the request cannot be met.
template <int V, int RI>
int blocks_per_sm_vr(size_t smem) {
  int nb0 = 0, nb1 = 0;
  if (cudaFuncSetAttribute(pair_kernel<V, false, RI>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) !=
          cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb0, pair_kernel<V, false, RI>, kTile / RI, smem) !=
          cudaSuccess ||
      cudaFuncSetAttribute(pair_kernel<V, true, RI>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) !=
          cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb1, pair_kernel<V, true, RI>, kTile / RI, smem) !=
          cudaSuccess) {
    (void)cudaGetLastError();
    return 0;
  }
  return nb0 < nb1 ? nb0 : nb1;
}

template <int V>
int blocks_per_sm_v(int hist_width, int depth, int block) {
  size_t smem = pair_kernel_smem(hist_width, depth, block);
  if (block == kBlockSmall) {  // the aggregated-increment instance must fit as well
    int na = 0;
    if (cudaFuncSetAttribute(pair_kernel<V, false, 4, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) !=
            cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&na, pair_kernel<V, false, 4, true>, kBlockSmall, smem) !=
            cudaSuccess) {
      (void)cudaGetLastError();
      return 0;
    }
    const int nb = blocks_per_sm_vr<V, 4>(smem);
    return na < nb ? na : nb;
  }
  return block == kBlockHuge ? blocks_per_sm_vr<V, 1>(smem)
         : block == kBlockLarge ? blocks_per_sm_vr<V, 2>(smem) : blocks_per_sm_vr<V, 4>(smem);
}

int pair_kernel_blocks_per_sm(int variant, int hist_width, int depth, int block) {
  switch (variant) {
    case V_NONE: return blocks_per_sm_v<V_NONE>(hist_width, depth, block);
    case V_ORTHO: return blocks_per_sm_v<V_ORTHO>(hist_width, depth, block);
    case V_TRIC: return blocks_per_sm_v<V_TRIC>(hist_width, depth, block);
    default: return blocks_per_sm_v<V_TRIC_SEARCH>(hist_width, depth, block);
  }
}

cudaError_t launch_stage(const StageJob* jobs, int n_jobs, int64_t n_chunks, cudaStream_t stream) {
  clear_stale_error();
  if (n_jobs <= 0 || n_chunks <= 0) return cudaSuccess;
  stage_kernel<<<(unsigned)n_chunks, 256, 0, stream>>>(jobs, n_jobs);
  return cudaGetLastError();
}

cudaError_t launch_spatial_sort(const SortSeg* segs, int n_segs, const SortPlan& plan, const float4* src, float4* dst,
                                const double4* src64, double4* dst64, int2* keys, uint32_t* counts,
                                cudaStream_t stream) {
  clear_stale_error();
  if (n_segs <= 0 || plan.chunks <= 0) return cudaSuccess;
  uint32_t* const cursors = counts + plan.keys;
  const unsigned chunks = (unsigned)plan.chunks;
  for (int pass = 0; pass < 3; ++pass) {
    if (plan.tiles[pass] == 0) continue;
    sort_count_kernel<<<chunks, 256, 0, stream>>>(segs, n_segs, pass, src, keys, counts, cursors);
    sort_scan_kernel<<<(unsigned)plan.tiles[pass], 1024, 0, stream>>>(segs, n_segs, pass, counts, cursors);
  }
  sort_scatter_kernel<<<chunks, 256, 0, stream>>>(segs, n_segs, src, src64, keys, cursors, dst, dst64);
  run_bounds_kernel<<<(unsigned)plan.bblocks, 32 * kBoundRuns, 0, stream>>>(segs, n_segs);
  return cudaGetLastError();
}

cudaError_t launch_prep(const StageJob* jobs, int n_jobs, int64_t max_n, bool strips, const SortSeg* sorts,
                        uint32_t* counts, cudaStream_t stream) {
  clear_stale_error();
  if (n_jobs <= 0) return cudaSuccess;
  const unsigned blocks = (unsigned)prep_blocks(max_n);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(blocks * (unsigned)n_jobs);
  cfg.blockDim = dim3(kPrepBlock);
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = blocks;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (max_n * 2 > kPrepMaxN) return cudaLaunchKernelEx(&cfg, prep_kernel<8, true>, jobs, sorts, counts);
  return strips ? cudaLaunchKernelEx(&cfg, prep_kernel<4, true>, jobs, sorts, counts)
                : cudaLaunchKernelEx(&cfg, prep_kernel<4, false>, jobs, sorts, counts);
}

cudaError_t launch_frame_setup(FrameDev* frames, int n_frames, bool order, bool windows, cudaStream_t stream) {
  clear_stale_error();
  if (n_frames <= 0) return cudaSuccess;
  frame_setup_kernel<<<n_frames, 128, 0, stream>>>(frames, order, windows);
  return cudaGetLastError();
}

cudaError_t launch_thresholds(double r_max, int32_t nbins, double* T, int32_t* status,
                              cudaStream_t stream) {
  clear_stale_error();
  int threads = 128;
  int blocks = (nbins + 1 + threads - 1) / threads;
  thresholds_kernel<<<blocks, threads, 0, stream>>>(r_max, nbins, T, status);
  return cudaGetLastError();
}

template <int V, bool MULTI, int RI, bool AGG = false>
cudaError_t launch_pairs_vmr(const PairLaunch& p, int grid, size_t smem, cudaStream_t stream) {
  clear_stale_error();
  cudaError_t e =
      cudaFuncSetAttribute(pair_kernel<V, MULTI, RI, AGG>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  pair_kernel<V, MULTI, RI, AGG><<<grid, kTile / RI, smem, stream>>>(p);
  return cudaGetLastError();
}

template <int V, bool MULTI>
cudaError_t launch_pairs_vm(const PairLaunch& p, int grid, size_t smem, cudaStream_t stream) {
  if constexpr (!MULTI)  // aggregated increments: 256-thread blocks, one sweep
    if (p.agg && (p.block == kBlockSmall || p.block == 0)) return launch_pairs_vmr<V, false, 4, true>(p, grid, smem, stream);
  return p.block == kBlockHuge    ? launch_pairs_vmr<V, MULTI, 1>(p, grid, smem, stream)
         : p.block == kBlockLarge ? launch_pairs_vmr<V, MULTI, 2>(p, grid, smem, stream)
                                  : launch_pairs_vmr<V, MULTI, 4>(p, grid, smem, stream);
}

template <int V>
cudaError_t launch_pairs_v(const PairLaunch& p, int grid, size_t smem, cudaStream_t stream) {
  return p.multi ? launch_pairs_vm<V, true>(p, grid, smem, stream) : launch_pairs_vm<V, false>(p, grid, smem, stream);
}

cudaError_t launch_pairs(const PairLaunch& p, int variant, int grid, size_t smem, cudaStream_t stream) {
  switch (variant) {
    case V_NONE: return launch_pairs_v<V_NONE>(p, grid, smem, stream);
    case V_ORTHO: return launch_pairs_v<V_ORTHO>(p, grid, smem, stream);
    case V_TRIC: return launch_pairs_v<V_TRIC>(p, grid, smem, stream);
    default: return launch_pairs_v<V_TRIC_SEARCH>(p, grid, smem, stream);
  }
}

}  // namespace dh
