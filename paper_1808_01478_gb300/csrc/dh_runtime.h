// Host-runtime internals shared by the plain/batched path (dh_runtime.cpp) and
// the served path (dh_serve.cpp).  Not part of the public ABI.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>
#include <map>
#include <memory>
#include <mutex>
#include <string>
#include <unordered_map>
#include <vector>

#include "../../include/dh.h"
#include "dh_internal.h"

namespace dh {

// Record a failure message for dh_last_error() on this thread and return s.
dh_status fail(dh_status s, const char* fmt, ...);
const char* last_error_message();

#define DH_CUDA_TRY(expr)                                                                        \
  do {                                                                                           \
    cudaError_t e_ = (expr);                                                                     \
    if (e_ != cudaSuccess)                                                                       \
      return ::dh::fail(e_ == cudaErrorMemoryAllocation ? DH_ERR_NOMEM : DH_ERR_CUDA, "%s: %s", \
                        #expr, cudaGetErrorString(e_));                                          \
  } while (0)

// Device buffer that only grows.
struct DevBuf {
  void* p = nullptr;
  size_t cap = 0;
  cudaError_t ensure(size_t bytes);
  void release();
};

// Pinned host buffer that only grows.
struct HostBuf {
  void* p = nullptr;
  size_t cap = 0;
  cudaError_t ensure(size_t bytes);
  void release();
};

// Binary64 bin-threshold tables per (r_max, nbins), shared by all paths of a
// context.  acquire() returns a table (building it on `st` if missing) and
// holds a reference; release() drops it.  A table built on one stream is made
// visible to work on another stream through an event wait.  Unreferenced tables
// beyond the cap are freed stream-ordered.
class ThresholdCache {
 public:
  dh_status acquire(double r_max, int32_t nbins, cudaStream_t st, int32_t* status_dev, double** T,
                    int* launched);
  void release(const double* T);
  void clear(cudaStream_t st);

 private:
  struct Key {
    uint64_t rbits;
    int32_t nbins;
    bool operator<(const Key& o) const { return rbits != o.rbits ? rbits < o.rbits : nbins < o.nbins; }
  };
  struct Entry {
    double* T;
    int refs;
    uint64_t last;
    cudaStream_t built_on;  // stream of the build kernel
    cudaEvent_t ready;      // recorded after it; other streams wait on it
  };
  std::mutex mu_;
  std::map<Key, Entry> map_;
  std::unordered_map<const double*, Key> rev_;
  uint64_t tick_ = 0;
  size_t cap_ = 64;
};

// A frame checked and planned on the host.
struct PlannedFrame {
  const dh_frame* src;
  int32_t variant;
  int32_t n_hist;
  int32_t sweeps;
  int32_t sweep_width;
  double margin;
  uint64_t pairs;
  bool list;  // the list kernel can run it,
  bool pick;  //   with the shortest of several images of a pair inside r_max
};

// list_width: bins per sweep of the list kernel, 0 when the caller has no list path.
dh_status check_frame(const dh_frame* f, PlannedFrame& pf, int max_width, int list_width);
void fill_frame_dev(const PlannedFrame& pf, FrameDev& F, const float4* X, uint64_t* out, const double* T);
// jm: j tiles of kTile/jm particles per i tile of kTile.  fill_segments writes
// at most cap segments to out and the total to *n_out; add_segments appends all.
int64_t fill_segments(const PlannedFrame& pf, FrameDev* fd, int64_t item0, int jm, Segment* out, int cap,
                      int* n_out);
int64_t add_segments(const PlannedFrame& pf, FrameDev* fd, int64_t item0, std::vector<Segment>& segs, int jm = 1);

// The same for the list kernel: split items per run pair, more (up to 16) in segments
// that would have fewer than `least` items, kListLeast for two per warp of a block.
constexpr int kListLeast = 2 * kListBlock / 32;
int64_t add_list_segments(const PlannedFrame& pf, FrameDev* fd, int64_t item0, std::vector<ListSegment>& segs,
                          int split, int least);
// Orders the segments of one list-kernel launch of `grid` blocks for its work distribution
// and fills L's n_segs, n_shared, shared_blocks, n_items and shared_items.  A segment
// of at most a 32nd of a block's share of the launch is one block's own: the blocks
// take these in order from one counter, and the last of them can keep a block no longer
// than a 32nd of its time past the others (an eighth: 2,000 frames of 2,000 particles
// 8.4 -> 8.6 ms, served requests of mixed sizes 6.03 -> 6.20 ms).
void list_share_segments(ListSegment* segs, size_t n, int grid, ListLaunch& L);
int64_t frame_runs(const dh_frame* f);  // runs of kRun particles over its species
// Estimated time of a frame's species pairs in a launch that fills `num_sms` SMs, in
// microseconds, on the list kernel and on the tiled kernel, and of the latter's longest item.
//
// The list kernel evaluates a particle's images against whole runs of 128, whose boxes are
// large parts of the cell when a species is small: of the cell's volume, a box with sides f
// widened by r_max = rho cells all around takes V = f^3 + 6 f^2 rho + 3 pi f rho^2 + 4/3 pi rho^3,
// as many pairs per pair of particles (6.9 for species of one run and rho = 1/2; a quarter
// more in a skewed cell).  The tiled
// kernel evaluates every pair once, in whole tiles.  So a species pair takes
//   list:  9 us (20 with a box) + 0.11 ns V per pair, padded to runs,
//   tiled: 2.5 us + 0.125 ns per pair of its tiles; a tile 24 us + 0.13 ns per pair on its own.
// Where the shortest of several images counts (PlannedFrame.pick), particles with more than
// one candidate are evaluated image by image: 0.1 + 2.4 f ns per pair on the list kernel,
// times V where r_max holds only a part of the cell.  Orthorhombic, r_max = 0.85 L,
// N = 40,000: list 2.27 ms, tiled 0.66; N = 500,000: 185 and 69 ms; a rod of 1 : 1 : 50, N =
// 200,000: 144 and 11.5 ms; N = 1,500: 43 and 160 us; r_max = 0.75 of the short side of a
// 1 : 10 : 10 slab, N = 200,000: 2.2 and 2.6 ms.
// All fitted to calls of 1 to 3,000 frames of 100 to 12,000 particles in 1 to 100 species, of all
// box types, which they meet within a third.  N = 1,500 in 8 species, orthorhombic, 1,777
// frames: list 22.6 ms, tiled 4.4 ms; N = 6,000 in one species, 111 frames: 1.85 and 1.88 ms;
// N = 12,000 in 3, 27 frames: 2.05 and 1.67 ms, with r_max a third of that half as much as tiled.
struct FrameCost {
  double list = 0.0, tiled = 0.0, tile = 0.0;
};
FrameCost frame_cost(const PlannedFrame& pf, int num_sms);
// Frames that may choose: the tiled kernel takes the 27-image search several times slower.
inline bool may_be_tiled(const PlannedFrame& pf) { return pf.list && pf.variant != V_TRIC_SEARCH; }
// Marks the frames of a call for which the tiled kernel is worth its launch, its setup and
// the wait for its last tile (costs: of the frames that may choose; n of all others).
bool choose_tiled(const std::vector<FrameCost>& costs, size_t others, std::vector<char>* tiled);
// Items per run pair: one item per warp where the frames are that small, else
// enough for an even end.
int list_split_for(double run_pairs, int num_sms);

// Launch shape of one pair-kernel launch.
struct LaunchParams {
  int32_t list = 0;              // the list kernel (the fields below do not apply)
  int32_t jm = 1;                // j tiles per i tile: tile_j = kTile / jm
  int32_t depth = 1;             // private histogram copies per block
  int32_t bps = 0;               // blocks per SM (0: as many as fit)
  int32_t block = kBlockSmall;   // threads per block (kBlockSmall, kBlockLarge or kBlockHuge)
  int32_t agg = 0;               // 256-thread blocks, one sweep: warp-aggregated increments
};

// Autotuner key of a launch: variant, histogram width, frame size, frame count (all bucketed).
struct TuneKey {
  int32_t variant = 0, width_log2 = 0, n_log2 = 0, frames_log4 = 0;
  bool operator<(const TuneKey& o) const {
    if (variant != o.variant) return variant < o.variant;
    if (width_log2 != o.width_log2) return width_log2 < o.width_log2;
    if (n_log2 != o.n_log2) return n_log2 < o.n_log2;
    return frames_log4 < o.frames_log4;
  }
};
struct TuneEntry {
  LaunchParams p;
  double gpairs_s = 0.0;
  bool old = false;  // measured before there was a list kernel to compare with: counted, but not used
};
TuneKey make_tune_key(int variant, int width, double mean_pairs_per_frame, int frames);

// Bytes of a frame's coordinate array (float32 or binary64, 3 or 4 per particle).
size_t coord_bytes(const dh_frame* f);

// Species are put in spatial order before the pair kernel, over the frame's
// bounding box or its home cell (SortSeg).  plan_spatial_order lists the species of
// one frame (its particles from x0 in the packed coordinates, its counters from
// key0); not for the list kernel, frames of the search and those of species below
// kSortMinTiled keep their order.
// list: the list kernel runs the frame, and its larger species are ordered in strips.
std::vector<SortSeg> plan_spatial_order(const PlannedFrame& pf, bool list, const FrameDev* fd, int64_t x0, int64_t key0,
                                        SortPlan* plan);
// Strips instead of the Hilbert curve: the runs' boxes are smaller, so that fewer pairs
// beyond r_max are evaluated and fewer pairs re-decided (whole call, orthorhombic
// N = 32,000 422 -> 406 us, N = 100,000 2.43 -> 2.27 ms, pair kernel at N = 1,000,000
// 170.2 -> 162.4 ms; N = 200,000 with 100,000 bins 15.8 -> 14.2 ms), for two passes more
// (10 us in launch_prep, 20 as kernels): at N = 16,000 188 against 182 us triclinic and
// 190 against 191 orthorhombic, at N = 12,000 144 against 153.  Without a box nothing is
// gained where r_max holds the whole frame: N = 60,000 1.01 against 1.03 ms, from
// N = 200,000 on even.  Species of a few runs have nothing to gain either way.
constexpr int64_t kSortMinTiled = 2048;
constexpr int64_t kStripMinN = 16000, kStripMinNoBoxN = 200000, kStripMinSpecies = 2048;

// Threads per block for a launch without a measured shape: from 16,384 bins on,
// a 256-thread block's histogram leaves room for at most two blocks per SM, and
// one 1024-thread block sharing one histogram keeps more warps resident (512
// threads when the larger block's queues do not fit next to the histogram).
int default_block(int variant, int width);

// Measured launch shapes per key (dh_tune.cpp), optionally kept in a text file.
class Tuner {
 public:
  bool lookup(const TuneKey& k, LaunchParams* p);
  void store(const TuneKey& k, const TuneEntry& e);
  size_t size();
  int load(const std::string& path, int sms);   // entries read, -1 if the file cannot be read
  bool save(const std::string& path, int sms);

 private:
  std::mutex mu_;
  std::map<TuneKey, TuneEntry> map_;
};
// Blocks for the pair kernel: `bps` per SM, at most one per item.
int pair_grid(int num_sms, int bps, int64_t n_items);

class Server;  // served path (dh_serve.cpp)
Server* server_create(dh_ctx* c, dh_status* st);
void server_destroy(Server* s);
dh_status server_submit(Server* s, const dh_frame* f, uint64_t* ticket);
dh_status server_poll(Server* s, uint64_t ticket);
dh_status server_wait(Server* s, uint64_t ticket, uint64_t timeout_ns);
dh_status server_cancel(Server* s, uint64_t ticket);

}  // namespace dh

struct dh_ctx {
  int device = 0;
  cudaStream_t own_stream = nullptr;
  cudaStream_t user_stream = nullptr;
  bool has_user_stream = false;
  std::recursive_mutex mu;
  int num_sms = 0;
  int max_width = 0;
  int list_width = 0;
  dh_config cfg{};

  dh::DevBuf raw;      // caller coordinates copied from the host (n x stride floats)
  dh::DevBuf X;        // packed float4 coordinates
  dh::DevBuf hist;     // uint64 histograms (host-pointer outputs)
  dh::DevBuf meta;     // FrameDev | StageJob | Segment arrays
  dh::DevBuf ctl;      // Control
  dh::HostBuf hmeta;   // pinned staging for meta
  dh::HostBuf hout;    // pinned staging for accumulate-on-host
  dh::DevBuf tstat;    // threshold build status,
  bool tstat_new = false;  //   to be read after the call: a table was built
  dh::DevBuf aux;      // small per-call arrays (g(r) pair densities)
  dh::DevBuf X64;      // binary64 input coordinates (double4), when a frame has them
  dh::DevBuf P4, P2;   // list kernel: positions in bins (double-floats),
  dh::DevBuf bnd;      //   bounds of the runs
  dh::DevBuf sortX64;  // staged in the caller's order: binary64,
  dh::DevBuf sortX;    // and float32 coordinates,
  dh::DevBuf sortK;    //   each particle's cell and place in it,
  dh::DevBuf sortC;    //   and cell counters
  dh::ThresholdCache tcache;
  std::vector<const double*> held_tables;  // tables referenced by work not yet finished

  dh::Tuner tuner;
  std::string tune_path;           // autotuner cache file ("" for none)
  bool tune_forced = false;        // measurement in progress: every launch uses tune_force
  dh::LaunchParams tune_force;
  int32_t tune_runs = 0;           // measurement launches made for the current call
  double tune_cap_pairs = 0.0;     // measurement: stop each pair-kernel launch after about this many pairs

  dh_stats stats{};
  cudaEvent_t ev_pair0 = nullptr, ev_pair1 = nullptr;  // pair-kernel timing (DH_CFG_TIMING)
  bool timed = false;
  bool pending_async = false;
  // of the last asynchronous call: its descriptors are uploaded (the pinned copy may be
  // written again), and all of it is done (the workspace may be used on another stream)
  cudaEvent_t ev_meta = nullptr, ev_async = nullptr;
  bool async_in_flight = false;
  cudaGraphExec_t gexec = nullptr;  // batched path: executable graph, updated per call

  std::mutex server_mu;
  dh::Server* server = nullptr;

  cudaStream_t stream() const { return has_user_stream ? user_stream : own_stream; }
};
