// dh_histogram_noalloc: the histogram of one frame without allocating memory.
//
// The regular entry points keep their workspace (packed coordinates, the
// binary64 threshold table, frame and work descriptors, the work counter) in
// device memory that the context allocates with cudaMalloc on first use.  Some
// callers cannot allow that: code inside a framework whose device memory is
// owned by its own allocator (a cudaMalloc behind its back fragments or
// overcommits the pool it manages), or a process that runs under a fixed
// device-memory budget, must not trigger new device allocations.  This variant
// takes device input and output from the
// caller and keeps all of its scratch in one file-scope __device__ array of a
// fixed size, so it never calls cudaMalloc, cudaFree or any other allocating
// routine.  The paper has no counterpart of it.
//
// The array is reserved on every GPU that loads the library and is kept until
// the process exits.  All calls share it: a call clears what must start at
// zero, and calls whose GPU work overlaps (different streams, host threads or
// processes sharing one context) race on it.
#include <cuda_runtime.h>

#include <cstring>
#include <mutex>
#include <new>
#include <vector>

#include "dh_runtime.h"

namespace dh {
namespace {

// Scratch layout (bytes, each part 256-byte aligned).
constexpr size_t kNaCtl = 256;                                  // Control
constexpr size_t kNaFrame = 2048;                               // FrameDev
constexpr size_t kNaJob = 256;                                  // StageJob
constexpr size_t kNaSegs = 16 * 1024;                           // Segment[] (256 of them)
constexpr size_t kNaT = ((size_t)DH_NOALLOC_MAX_BINS + 1) * 16; // thresholds + float-pair copy
constexpr size_t kNaTPad = (kNaT + 255) & ~(size_t)255;
constexpr size_t kNaX = (size_t)DH_NOALLOC_MAX_N * 16;          // float4 coordinates
constexpr size_t kNaOffFrame = kNaCtl;
constexpr size_t kNaOffJob = kNaOffFrame + kNaFrame;
constexpr size_t kNaOffSegs = kNaOffJob + kNaJob;
constexpr size_t kNaOffT = kNaOffSegs + kNaSegs;
constexpr size_t kNaOffX = kNaOffT + kNaTPad;
constexpr size_t kNaBytes = kNaOffX + kNaX;
static_assert(kNaBytes == DH_NOALLOC_SCRATCH_BYTES, "scratch size must match the value published in dh.h");
static_assert(sizeof(FrameDev) <= kNaFrame && sizeof(StageJob) <= kNaJob && sizeof(Control) <= kNaCtl,
              "scratch slots too small");
constexpr int kNaMaxSegs = (int)(kNaSegs / sizeof(Segment));
constexpr int kNaMaxDevices = 64;

// Frames of the list kernel share the scratch out anew, in one upload up to T:
//   Control | FrameDev | StageJob | SortSeg[] | ListSegment[] | SegCounter[] |
//   T | run bounds | P4 | P2 | ordered coordinates | cell counters
// (about 46 bytes per particle and 16 per bin: 60,000 particles with 10,000 bins).
struct NaListPlan {
  PlannedFrame pf;
  std::vector<SortSeg> sorts;
  std::vector<ListSegment> segs;
  int64_t items = 0;
  int split = 1, strips = 0, grid = 0;
  ListLaunch launch;
  size_t sort_at = 0, seg_at = 0, ctr_at = 0, T_at = 0, bnd_at = 0, P4_at = 0, P2_at = 0, X_at = 0, cells_at = 0;
};

// False when the frame is not one for the list kernel or does not fit: the tiled kernel takes it.
bool plan_list(const dh_frame* f, int max_width, int num_sms, unsigned char* base, NaListPlan& p) {
  if (check_frame(f, p.pf, max_width, list_kernel_max_width()) != DH_OK || !p.pf.list) return false;
  std::vector<char> tiled;
  if (may_be_tiled(p.pf) && choose_tiled({frame_cost(p.pf, num_sms)}, 0, &tiled)) return false;
  FrameDev* fd = (FrameDev*)(base + kNaOffFrame);
  SortPlan sort;
  p.sorts = plan_spatial_order(p.pf, true, fd, 0, 0, &sort);
  p.strips = sort.max_keys[0] > 0;
  if (!prep_fits(f->n, sort.keys)) return false;
  p.split = list_split_for((double)p.pf.pairs / ((double)kRun * kRun) * p.pf.sweeps, num_sms);
  p.items = add_list_segments(p.pf, fd, 0, p.segs, p.split, kListLeast);
  p.grid = pair_grid(num_sms, 1, p.items);
  std::memset(&p.launch, 0, sizeof p.launch);
  list_share_segments(p.segs.data(), p.segs.size(), p.grid, p.launch);
  size_t at = kNaOffSegs;
  auto part = [&at](size_t bytes) {
    const size_t here = at;
    at += (bytes + 255) & ~(size_t)255;
    return here;
  };
  p.sort_at = part(sizeof(SortSeg) * p.sorts.size());
  p.seg_at = part(sizeof(ListSegment) * p.segs.size());
  p.ctr_at = part(sizeof(SegCounter) * ((size_t)p.launch.n_shared + 1));
  p.T_at = part(16 * ((size_t)f->nbins + 1));
  p.bnd_at = part(2 * sizeof(float4) * (size_t)frame_runs(f));
  p.P4_at = part(sizeof(float4) * (size_t)f->n);
  p.P2_at = part(sizeof(float2) * (size_t)f->n);
  p.X_at = part(sizeof(float4) * (size_t)f->n);
  p.cells_at = part(sizeof(uint32_t) * (size_t)sort.keys);
  return at <= kNaBytes;
}

// The scratch itself.  Host code must not pass this name to a kernel: on the
// host it is only a stand-in; its device address comes from cudaGetSymbolAddress.
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNaBytes];

std::mutex g_na_mu;
unsigned char* g_na_ptr[kNaMaxDevices] = {};

// Device address of the scratch on the current device, looked up once per device.
dh_status scratch_for_current_device(unsigned char** out) {
  int dev = -1;
  DH_CUDA_TRY(cudaGetDevice(&dev));
  if (dev < 0 || dev >= kNaMaxDevices) return fail(DH_ERR_INVALID, "device %d out of range", dev);
  std::lock_guard<std::mutex> g(g_na_mu);
  if (!g_na_ptr[dev]) {
    void* p = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e != cudaSuccess || !p)
      return fail(DH_ERR_CUDA, "cudaGetSymbolAddress(scratch): %s", cudaGetErrorString(e));
    g_na_ptr[dev] = (unsigned char*)p;
  }
  *out = g_na_ptr[dev];
  return DH_OK;
}

}  // namespace
}  // namespace dh

using namespace dh;

static dh_status histogram_noalloc(const dh_frame* frame, void* stream_ptr) {
  if (!frame) return fail(DH_ERR_INVALID, "frame is NULL");
  if (!(frame->flags & DH_DEVICE_PTRS))
    return fail(DH_ERR_INVALID, "dh_histogram_noalloc needs DH_DEVICE_PTRS (device coords and out)");
  if (frame->flags & DH_COORDS_F64)
    return fail(DH_ERR_INVALID, "dh_histogram_noalloc takes float32 coordinates");
  if (frame->n > DH_NOALLOC_MAX_N)
    return fail(DH_ERR_INVALID, "n = %lld exceeds the allocation-free limit of %d particles",
                (long long)frame->n, DH_NOALLOC_MAX_N);
  if (frame->nbins > DH_NOALLOC_MAX_BINS)
    return fail(DH_ERR_INVALID, "nbins = %d exceeds the allocation-free limit of %d bins", frame->nbins,
                DH_NOALLOC_MAX_BINS);
  int dev = -1;
  DH_CUDA_TRY(cudaGetDevice(&dev));
  int num_sms = 0, max_width = 0;
  DH_CUDA_TRY(cudaDeviceGetAttribute(&num_sms, cudaDevAttrMultiProcessorCount, dev));
  max_width = pair_kernel_max_width();
  if (max_width < 1024) return fail(DH_ERR_CUDA, "not enough shared memory per block");
  PlannedFrame pf;
  dh_status s = check_frame(frame, pf, max_width, 0);
  if (s != DH_OK) return s;
  unsigned char* base = nullptr;
  s = scratch_for_current_device(&base);
  if (s != DH_OK) return s;
  cudaStream_t st = (cudaStream_t)stream_ptr;

  Control* ctl = (Control*)(base);
  FrameDev* fd = (FrameDev*)(base + kNaOffFrame);
  StageJob* job = (StageJob*)(base + kNaOffJob);
  Segment* segs = (Segment*)(base + kNaOffSegs);

  // Every host-side check comes before the first enqueued operation, so that a
  // call that fails leaves the caller's output and the shared scratch untouched.
  Segment hS[kNaMaxSegs];
  int n_segs = 0;
  const int64_t n_items = fill_segments(pf, fd, 0, 1, hS, kNaMaxSegs, &n_segs);
  if (n_segs > kNaMaxSegs)
    return fail(DH_ERR_INVALID, "%d species x %d sweeps need %d work segments, beyond the allocation-free limit of %d",
                frame->n_species, pf.sweeps, n_segs, kNaMaxSegs);
  const int block = default_block(pf.variant, pf.sweep_width);
  const int bps = n_items > 0 ? pair_kernel_blocks_per_sm(pf.variant, pf.sweep_width, 1, block) : 1;
  if (bps < 1) return fail(DH_ERR_INVALID, "histogram of %d bins does not fit in shared memory", pf.sweep_width);

  // Small frames go the way of dh_histogram: ordered by launch_prep and counted by
  // the list kernel (N = 30,000 triclinic, two species, 8,192 bins: 595 -> 389 us).
  NaListPlan lp;
  const bool list = plan_list(frame, max_width, num_sms, base, lp);
  double* T = (double*)(base + (list ? lp.T_at : kNaOffT));
  float4* X = (float4*)(base + (list ? lp.X_at : kNaOffX));
  const bool clear = !(frame->flags & DH_ACCUMULATE);
  const size_t out_words = (size_t)pf.n_hist * (size_t)frame->nbins;
  const bool prep_clear = list && clear && (int64_t)out_words <= prep_clears(frame->n);

  // The descriptors, uploaded in one copy that has read them when it returns; what
  // must start at zero is part of it.
  std::vector<unsigned char> up(list ? lp.T_at : kNaOffSegs + sizeof(Segment) * (size_t)n_segs, 0);
  FrameDev& hF = *(FrameDev*)(up.data() + kNaOffFrame);
  fill_frame_dev(list ? lp.pf : pf, hF, X, frame->out, T);
  StageJob& hJ = *(StageJob*)(up.data() + kNaOffJob);
  hJ.src = frame->coords;
  hJ.dst = X;
  hJ.fd = fd;
  hJ.n = frame->n;
  hJ.stride = (frame->flags & DH_COORDS_F4) ? 4 : 3;
  if (list) {
    hF.bnd = (float4*)(base + lp.bnd_at);
    hF.P4 = (float4*)(base + lp.P4_at);
    hF.P2 = (float2*)(base + lp.P2_at);
    hJ.n_sort = (int32_t)lp.sorts.size();
    hJ.strips = lp.strips;
    hJ.clear = prep_clear ? (int64_t)out_words : 0;
    std::memcpy(up.data() + lp.sort_at, lp.sorts.data(), sizeof(SortSeg) * lp.sorts.size());
    if (!lp.segs.empty()) std::memcpy(up.data() + lp.seg_at, lp.segs.data(), sizeof(ListSegment) * lp.segs.size());
  } else if (n_segs > 0) {
    std::memcpy(up.data() + kNaOffSegs, hS, sizeof(Segment) * (size_t)n_segs);
  }
  DH_CUDA_TRY(cudaMemcpyAsync(base, up.data(), up.size(), cudaMemcpyHostToDevice, st));
  DH_CUDA_TRY(launch_thresholds(frame->r_max, frame->nbins, T, &ctl->status, st));
  if (clear && !prep_clear) DH_CUDA_TRY(cudaMemsetAsync(frame->out, 0, sizeof(uint64_t) * out_words, st));
  if (list) {
    DH_CUDA_TRY(launch_prep(job, 1, frame->n, lp.strips != 0, (const SortSeg*)(base + lp.sort_at), (uint32_t*)(base + lp.cells_at), st));
    if (lp.items > 0) {
      ListLaunch L = lp.launch;
      L.segs = (const ListSegment*)(base + lp.seg_at);
      L.ctr = (SegCounter*)(base + lp.ctr_at);
      L.hist_width = lp.pf.sweep_width;
      L.multi = lp.pf.sweeps > 1;
      L.pick = lp.pf.pick;
      DH_CUDA_TRY(launch_list(L, lp.grid, st));
    }
  } else {
    int64_t chunks = (frame->n + kStageChunk - 1) / kStageChunk;
    if (chunks > 0) DH_CUDA_TRY(launch_stage(job, 1, chunks, st));
    DH_CUDA_TRY(launch_frame_setup(fd, 1, false, false, st));
    if (n_items > 0) {
      PairLaunch L;
      std::memset(&L, 0, sizeof L);
      L.block = block;
      L.segs = segs;
      L.n_segs = n_segs;
      L.n_items = n_items;
      L.hist_width = pf.sweep_width;
      L.multi = pf.sweeps > 1;
      L.ctl = ctl;
      DH_CUDA_TRY(launch_pairs(L, pf.variant, pair_grid(num_sms, bps, n_items),
                               pair_kernel_smem(pf.sweep_width, 1, block), st));
    }
  }
  // Read back the flags (in Control and FrameDev) and wait.
  DH_CUDA_TRY(cudaMemcpyAsync(up.data(), base, kNaOffJob, cudaMemcpyDeviceToHost, st));
  DH_CUDA_TRY(cudaStreamSynchronize(st));
  if (((const Control*)up.data())->status != 0) return fail(DH_ERR_CUDA, "bin threshold table did not converge");
  if (hF.bad) return fail(DH_ERR_INVALID, "frame has non-finite coordinates");
  return DH_OK;
}

// (the descriptors are kept in host vectors, all of them made before the first enqueued operation)
extern "C" dh_status dh_histogram_noalloc(const dh_frame* frame, void* stream_ptr) {
  try {
    return histogram_noalloc(frame, stream_ptr);
  } catch (const std::bad_alloc&) {
    return DH_ERR_NOMEM;
  }
}
