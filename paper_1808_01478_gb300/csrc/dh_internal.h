// Internal interface between the host runtime (dh_runtime.cpp) and the CUDA
// kernels (dh_kernels.cu).  Not part of the public ABI.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace dh {

// Kernel variants of the minimum-image step (Eq. 5).
enum Variant : int32_t {
  V_NONE = 0,         // no periodic box
  V_ORTHO = 1,        // diagonal B: per-axis nearest image
  V_TRIC = 2,         // triclinic, r_max below half the smallest plane spacing: one wrap
  V_TRIC_SEARCH = 3,  // triclinic, larger r_max: Eq. 5 wrap plus the 27-image search
};

constexpr int kTile = 1024;          // i particles per work item (and the longest j tile)
constexpr int kSubJ = 256;           // j sub-chunk with its own tile image per warp
// Pair-kernel blocks: 256 threads with 4 i particles each, 512 with 2, or 1024 with 1.
constexpr int kBlockSmall = 256;
constexpr int kBlockLarge = 512;
constexpr int kBlockHuge = 1024;
constexpr int kQueueCap = 64;        // deferred pairs per warp queue
constexpr int kNumVariants = 4;
constexpr int kListBlock = 512;      // list kernel: threads per block, one block per SM
constexpr int kRun = 128;            // list kernel: consecutive particles of a species with one bounding box
constexpr int64_t kListMaxN = (int64_t)1 << 26;  // list kernel: particle and image index share 32 bits

// One frame as seen by the device.  Host fills the first part; the staging and
// setup kernels fill the second.
struct FrameDev {
  const float4* X;   // packed coordinates (x,y,z,0), frame-local index
  const double4* X64;  // binary64 input coordinates (x,y,z,0), or null for float32 input
  uint64_t* out;     // S(S+1)/2 x nbins histograms of this frame
  const double* T;   // binary64 thresholds T[0..nbins]
  const float2* Tf;  // the same thresholds as float pairs (hi, lo), hi + lo = T to ~2^-48
  int32_t variant;
  int32_t nbins;
  int32_t n;         // particles
  int32_t sweep_width;  // bins per sweep (pass p covers [p*w, min(nbins,(p+1)*w)))
  double r_max;
  double B[9];       // row-major, columns a,b,c
  double Linv[3];    // orthorhombic: 1.0/L per axis, binary64
  float Bf[9];       // float32 copies of B
  float Bl[9];       // float32(B - Bf): B as double-float (Bf + Bl)
  float invf[3];     // float32 reciprocals: ortho 1/Lx,1/Ly,1/Lz; triclinic 1/ax,1/by,1/cz
  float S;           // float32(nbins / r_max)
  float dr_f;        // float32(r_max / nbins), the bin width
  float rmax_f;      // float32(r_max)
  float S2;          // float32((nbins / r_max)^2)
  float margin;      // triclinic: 1 - 2 r_max / h_min (no-search precondition margin)
  float tshift[27][3];  // periodic images: -B k rounded once from binary64, k in {-1,0,1}^3
                        // (index 9 (kx+1) + 3 (ky+1) + (kz+1))
  float tserr[27][3];   // |tshift - (-B k)|, rounded up
  float convf[3];       // binary64 input: per-axis conversion error (conv), rounded up
  float kxdb;           // triclinic: largest |kx| times |ax32 - ax|, rounded up
  float dBf[9];         // |B32 - B| per entry, rounded up
  float tie_t[3];       // orthorhombic: t-space tie term of one wrapped axis (0: none), rounded up
  float tie_all;        // orthorhombic: the frame's tie term (all axes wrapped), rounded up
  float rr2;            // orthorhombic: (r_max (1 + 2/nbins))^2, rounded up
  double eps_S;      // |S - nbins/r_max| / (nbins/r_max)
  double eps_S2;     // |S2 - (nbins/r_max)^2| / (nbins/r_max)^2
  // ---- written on the device
  int32_t cmin[3];   // ordered-integer encodings of the per-axis coordinate min / max
  int32_t cmax[3];
  int32_t bad;       // a non-finite coordinate was seen
  int32_t all_defer; // float32 decisions are not safe for this frame: every pair is deferred
  int32_t in_range;  // no box, one sweep: every pair's root stays below nbins + 1 (the clamp is a no-op)
  int32_t cull_ok;   // no box: tiles can lie outside a sweep (several sweeps, or r_max below the extent)
  float beta_u;      // beta of tiles that take a uniform image (orthorhombic, triclinic)
  float beta_w[3];   // beta of tiles with a uniform image on all axes but a, wrapped per pair
  float tie_m[3];    // orthorhombic: margin of the uniform-image test (0: not needed)
  float mid2, mid1;  // double-float tier: |r2 - T[n]| <= mid2*r2 + mid1*s decides nothing
  float tie_eps;     // orthorhombic: | |d'_c| - L_c/2 | <= tie_eps is re-decided in binary64
  float delta;       // float32 window half-width in bin units at t = nbins (reported)
  float alpha_t, beta_t;  // the t-space bound alpha*t + beta behind the q-space test (per-pair images)
  float eps_s;       // search variant: fractional-coordinate ambiguity margin
  unsigned long long deferred;  // statistics: pairs queued for the double-float tier
  unsigned long long exact;     // pairs that also needed the binary64 replay
  unsigned long long uniform_pairs;  // pairs of (warp i run, j tile) blocks with one nearest image for all
  unsigned long long axis_pairs;     // pairs of such blocks whose image is uniform on all axes but one
  unsigned long long culled_pairs;   // pairs of blocks skipped: no pair of them has its bin in the sweep
  // ---- spatial order and list kernel (P4 null for other frames); lengths in bins:
  // S + S_l = nbins / r_max times the caller's.  From the host:
  float4* P4;         // home positions: x, y, z to a grid (list_grid) and the rest of x,
  float2* P2;         //   the rest of y and z
  float4* bnd;        // bounds of each run of kRun particles (two float4: min, max xyz; w of the
                      // first: 1 if some coordinate is beyond list_far)
  int32_t clear;      // words of output to clear in frame_setup_kernel (at most kSetupClears)
  const float4* staged;  // the coordinates before they are ordered (bulk_box; not in launch_prep)
  float S_l;          // nbins / r_max - S
  float img_h[27][3], img_l[27][3];  // image vectors -B k as double-floats (index as tshift)
  float period[3];    // a_x, b_y, c_z
  int32_t pick;       // r_max beyond half the distance between images: the shortest image counts
  // ... and from the device
  int32_t smin[3], smax[3];  // triclinic: range of the fractional coordinates, as cmin and cmax
  int32_t wrap;       // the coordinates span more than one cell: P4 is brought home to the first
                      // (1: in double-floats; 2: in binary64, from 4,096 cells on)
  int32_t list_slow;  // every pair in binary64 (no trust in the images, or distances beyond float32)
  int32_t list_all;   // every listed pair re-decided (window too wide)
  float key_lo[3], key_inv;  // spatial order: origin and inverse side of the grid
  float list_grid;    // grid of the positions' high parts (a power of two),
  float list_c0;      //   constant part of the window (see list_setup),
  float list_mid;     //   position error of the double-float tier,
  float cull_abs;     //   absolute slack of the distance bounds
  float list_far;     // no box: runs with a coordinate from here on (bins) are compared in binary64
};

// One species pair (a,b) of one frame and one bin sweep, cut into kTile x kTile
// work items numbered row by row over (ti, tj) (intra-species: tj >= ti only).
// A launch may carry only part of a segment's items: launch items
// [item0, item0 + count) are the segment's items [item_base, item_base + count).
struct Segment {
  FrameDev* fd;
  int32_t intra;     // a == b: only j tiles not below the i tile, pairs j > i
  int32_t h;         // histogram index within the frame
  int32_t pass;      // bin sweep: bins [pass*w, min(nbins, (pass+1)*w)), w = fd->sweep_width
  int32_t n_ti, n_tj;  // i tiles of kTile particles, j tiles of kTile/jm particles
  int32_t a0, na, b0, nb;  // frame-local particle ranges of species a and b
  int32_t jm;        // j tiles per i tile (1, 2 or 4; 0 means 1)
  int64_t item0;     // first launch item of this segment
  int64_t item_base; // segment-local index of that item
};

// The same for the list kernel: one species pair of one frame and one bin
// sweep as items of one run of kRun i particles against one run of j particles
// (or a part of it, split_log2), numbered row by row over (i run, j
// run); intra-species: j runs not below the i run.  The i side is the larger
// species.  Launch items [item0, item0 + items) are the segment's items from
// item_base on.
struct ListSegment {
  FrameDev* fd;
  int32_t intra, h, pass;
  int32_t n_ti, n_tj;      // runs of the i and the j species
  int32_t i0, ni, j0, nj;  // frame-local particle ranges
  int32_t i_run0, j_run0;  // their first runs in the frame's bounds
  int32_t split_log2;      // log2 of the items per run pair (0 to 4: kRun >> split_log2 j particles each)
  int64_t item0, item_base, items;
};

// Staging job: one frame's coordinates (n x stride floats) -> float4.
struct StageJob {
  const float* src;  // n x stride float32, or binary64 when dst64 is set
  float4* dst;
  double4* dst64;    // binary64 input: the values themselves (dst gets them rounded to float32)
  FrameDev* fd;
  int64_t n;
  int32_t stride;
  int32_t chunk0;    // first staging chunk of this job
  // launch_prep: the frame's species (SortSeg), and the words of its output to clear
  int32_t sort0, n_sort;
  int32_t strips, pad;  // some species is ordered in strips
  int64_t clear;
};
constexpr int kStageChunk = 1024;

// Spatial ordering of one species, by counting sorts whose cells are the keys; the
// histogram does not depend on the order of particles within a species.  Either in
// one pass along a Hilbert curve over 2^g cells per axis, which keeps any number of
// consecutive particles compact; or (nb > 0) in slabs of equal counts along x, each
// in columns along y, each along z, in three passes over cells of each axis: runs of
// kRun particles become boxes as near to cubes as can be.
struct SortSeg {
  const FrameDev* fd;
  int64_t x0;        // first particle (index into the packed coordinates)
  int64_t f0;        // x0 of the frame's first particle
  int64_t key0[3];   // first counter of each pass (Hilbert: of the last, the others have none)
  int32_t n;         // particles
  int32_t g;         // Hilbert: grid bits per axis
  int32_t nb[3];     // strips: cells along x, y and z, multiples of four
  int32_t n_slab, n_col;   // slabs, columns per slab
  int32_t slab, col;       // particles per slab and per column, multiples of kRun
  int32_t run0;      // first run of this species in the frame's bounds
  int32_t chunk0, tile0[3], bblock0;  // first block of the launches (number_sort_blocks)
};
// Counters of a pass.
__host__ __device__ inline int64_t sort_keys(const SortSeg& S, int pass) {
  if (S.nb[0] == 0) return pass < 2 ? 0 : S.g > 0 ? (int64_t)1 << (3 * S.g) : 4;
  return (int64_t)S.nb[pass] * (pass == 0 ? 1 : pass == 1 ? S.n_slab : S.n_slab * S.n_col);
}
constexpr int kSortChunk = 256;   // particles per block,
constexpr int kScanTile = 4096;   //   counters per block,
constexpr int kBoundRuns = 8;     //   runs per block of the order's launches

struct Control {
  unsigned long long next_item;  // dynamic work counter (reset before each launch)
  int32_t status;                // 0 ok, else an error code
  int32_t pad;
};

struct PairLaunch {
  const Segment* segs;
  int32_t n_segs;
  int32_t hist_width;  // shared-memory bins per histogram copy (the widest sweep of the launch)
  int64_t n_items;
  Control* ctl;
  int32_t hist_depth;  // private histogram copies per block (warp w uses copy w mod depth); 0 means 1
  int32_t multi;       // nonzero when some sweep of the launch starts above bin 0
  int32_t block;       // threads per block: kBlockSmall (0 means it), kBlockLarge or kBlockHuge
  int32_t agg;         // 256-thread blocks, one sweep: warp-aggregated histogram increments (match.any)
};

// Work counter of one shared segment of a list-kernel launch (zeroed before it), and
// after those one for the launch's own segments (next: segments handed out).
struct SegCounter {
  unsigned long long next;  // items claimed
  int32_t attached;         // blocks working on the segment
  int32_t pad;
};

struct ListLaunch {
  const ListSegment* segs;
  SegCounter* ctr;       // one per shared segment, and one
  int32_t n_segs;
  int32_t n_shared;      // the first n_shared segments are shared by blocks, each of the others
                         // is one block's own (list_share_segments)
  int32_t shared_blocks; // blocks that start on the shared ones
  int32_t hist_width;
  int64_t n_items, shared_items;
  int32_t multi;
  int32_t pick;          // frames whose pairs take the shortest of several images (FrameDev.pick)
};

// ---- launchers (dh_kernels.cu); all enqueue on `stream` and return the launch error
cudaError_t launch_stage(const StageJob* jobs, int n_jobs, int64_t n_chunks, cudaStream_t stream);
// Staging, setup and spatial order of small frames of the list kernel in one
// launch (jobs: one per frame, n <= max_n <= kPrepMaxN, dst and dst64 the ordered
// copies; strips: some species is ordered so; sorts: all their species; counts:
// their counters).
cudaError_t launch_prep(const StageJob* jobs, int n_jobs, int64_t max_n, bool strips, const SortSeg* sorts,
                        uint32_t* counts, cudaStream_t stream);
constexpr int64_t kPrepMaxN = 65536;
// Within reach of launch_prep: particles and counters of a frame.
constexpr int kPrepBlock = 1024, kPrepCluster = 8;
inline int prep_blocks(int64_t max_n) {
  // one particle per thread up to the largest portable cluster (two or four per
  // thread: N = 4,000 without a box 72 and 80 us a call instead of 65)
  int blocks = 1;
  while (blocks < kPrepCluster && (int64_t)blocks * kPrepBlock < max_n) blocks *= 2;
  return blocks;
}
// Words of output that launch_prep clears for a frame; a fill by the whole chip is the
// faster way beyond (a block clears 64 GB/s: one block and 67 MB, N = 1,000 in 20 species
// with 40,000 bins, 1.14 ms a call, with a fill 0.13 ms).
inline int64_t prep_clears(int64_t max_n) { return 16384 * (int64_t)prep_blocks(max_n); }
inline bool prep_fits(int64_t n, int64_t keys) {
  return n >= 1 && n <= kPrepMaxN && keys <= (int64_t)prep_blocks(n) * kPrepBlock * (2 * n <= kPrepMaxN ? 8 : 16);
}
// ... and better there than with the separate kernels, which use the whole chip.
constexpr int64_t kPrepBestN = 32768;
// order: the spatial order's grid and the list kernel's window too; windows: the tiled
// kernel's window also for frames of the list kernel.
constexpr int64_t kSetupClears = 65536;
cudaError_t launch_frame_setup(FrameDev* frames, int n_frames, bool order, bool windows, cudaStream_t stream);
// What a set of SortSeg needs.
struct SortPlan {
  int64_t keys = 0;               // counters of all passes
  int64_t max_keys[3] = {0, 0, 0};  // most counters of one in each pass
  int64_t chunks = 0, tiles[3] = {0, 0, 0}, bblocks = 0;  // blocks of the launches
  void add(const SortPlan& o) {
    keys += o.keys;
    for (int p = 0; p < 3; ++p) max_keys[p] = o.max_keys[p] > max_keys[p] ? o.max_keys[p] : max_keys[p];
  }
};
// Numbers the blocks of the segments' launches one after another, so that each block
// has work whatever the sizes, and any number of species fits a launch.
inline void number_sort_blocks(SortSeg* segs, size_t n, SortPlan& plan) {
  plan.chunks = plan.bblocks = 0;
  for (int64_t& t : plan.tiles) t = 0;
  for (size_t q = 0; q < n; ++q) {
    SortSeg& g = segs[q];
    g.chunk0 = (int32_t)plan.chunks;
    g.bblock0 = (int32_t)plan.bblocks;
    plan.chunks += (g.n + kSortChunk - 1) / kSortChunk;
    plan.bblocks += (g.n + (int64_t)kBoundRuns * kRun - 1) / ((int64_t)kBoundRuns * kRun);
    for (int p = 0; p < 3; ++p) {
      g.tile0[p] = (int32_t)plan.tiles[p];
      plan.tiles[p] += (sort_keys(g, p) + kScanTile - 1) / kScanTile;
    }
  }
}
// Orders each segment's particles from src (src64) into dst (dst64), and for the
// list kernel into the frame's P4 and P2 with the bounds of its runs.  counts:
// plan.keys counters, zeroed, then as many cursors; keys: two per particle; the
// binary64 arrays may be null.
cudaError_t launch_spatial_sort(const SortSeg* segs, int n_segs, const SortPlan& plan, const float4* src, float4* dst,
                                const double4* src64, double4* dst64, int2* keys, uint32_t* counts,
                                cudaStream_t stream);
cudaError_t launch_thresholds(double r_max, int32_t nbins, double* T, int32_t* status,
                              cudaStream_t stream);
// One pair-kernel launch over segments whose frames all have minimum-image variant `variant`.
cudaError_t launch_pairs(const PairLaunch& p, int variant, int grid, size_t smem, cudaStream_t stream);
// The list kernel (dh_list.cu): segments of any frames planned for it.
cudaError_t launch_list(const ListLaunch& p, int grid, cudaStream_t stream);
cudaError_t launch_check_list(const ListSegment* segs, int n_segs, uint64_t n_samples, uint64_t seed,
                              unsigned long long* out, cudaStream_t stream);
int list_kernel_max_width();  // widest sweep of the list kernel on the current device,
constexpr int kPickWords = 12288;  //   less these bins for frames that need the shortest image
cudaError_t launch_check_sqrt(unsigned long long* out, cudaStream_t stream);
cudaError_t launch_check_tiles(const FrameDev* F, int variant, uint64_t n_tiles, uint64_t seed,
                               unsigned long long* out, cudaStream_t stream);
cudaError_t launch_check_window(const FrameDev* F, uint64_t n_samples, uint64_t seed, unsigned long long* out,
                                cudaStream_t stream);
cudaError_t launch_rdf(const uint64_t* counts, int32_t n_hist, int32_t nbins, double r_max,
                       const double* pair_density, uint64_t n_frames, double* g, cudaStream_t stream);
size_t pair_kernel_smem(int hist_width, int depth = 1, int block = kBlockSmall);
int pair_kernel_max_width();
int pair_kernel_blocks_per_sm(int variant, int hist_width, int depth = 1, int block = kBlockSmall);

// Host/device shared definition of the binary64 bin of Alg. 1 (used to build thresholds).
int64_t host_bin_of(double r2, double r_max, int32_t nbins);
int build_thresholds_host(double r_max, int32_t nbins, double* T);

}  // namespace dh
