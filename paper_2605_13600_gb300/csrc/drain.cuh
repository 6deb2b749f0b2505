// drain.cuh -- the chunked batched uplift (drain.cu), driven by batch.cu.
#pragma once

#include <vector>

#include "scoup_internal.cuh"

namespace scoup {

// Pointers of one view part that are reset before a batch.
struct DrainViewInit {
  WsHeader* hdr;
  uint32_t* tile_count;
  uint32_t* tile_glob;
};

// Stream of one chunk lane, with the events that order its drain against
// staged region maps.
struct ChunkStreams {
  cudaStream_t ls;
  cudaEvent_t before_drain = nullptr;  // if set: the drain waits for it
  cudaEvent_t after_drain = nullptr;   // if set: recorded once the drain and merge are enqueued
};

// The drain's side of a view.
TileJob tile_job(const ViewJob& v, const LevelCodes& lc, float* accum, float* comp, WsHeader* scene_hdr, int C, int Crow);

// One chunk of nv <= kMaxDrainJobs views (HOST arrays, each view with a view
// part of its own): depth cut, projection and binning, one drain launch over
// every (view, tile) item, the same for the tiles open behind their cut, then
// the merge of the views' counters into their scenes' headers (api.cu).  ctr
// (DEVICE): the lane's two drain counters.
int run_chunk(const ViewJob* views, const TileJob* jobs, int nv, uint32_t* ctr, bool compensated, int warp_w,
              const ChunkStreams& cs);
// Resets view parts before their first use (headers, binning counters).
cudaError_t launch_view_init(const DrainViewInit* parts, int nparts, int max_tiles, cudaStream_t st);
// Adds each job's view counters into its scene header and clears them.
cudaError_t launch_view_merge(const TileJob* jobs, int njobs, cudaStream_t st);

// Device memory and the chunk schedule of the chunked form for one plan.
struct DrainLayout {
  int chunk = 0, lanes = 0, sample = -1;  // the configuration the layout was built for
  int max_tiles = 1;
  void* mem = nullptr;
  size_t bytes = 0;
  std::vector<UpliftWs> scene;         // per scene: its header and Morton-ordered copy
  std::vector<int32_t*> fci;           // per scene: codes cut to K entries (s > K) or null
  std::vector<float*> fcv;
  std::vector<UpliftWs> view;          // [lanes * chunk] view parts, each with its own header
  std::vector<ViewJob> views;          // chunk-major: [chunk_begin[c] .. chunk_begin[c + 1])
  std::vector<TileJob> jobs;           // as views
  std::vector<int> chunk_begin;        // [nchunks + 1]
  uint32_t* counters_dev = nullptr;    // [lanes][2]: the drain counters of each lane
  std::vector<DrainViewInit> init;     // [lanes * chunk]
};

// Builds (or rebuilds) the layout for `chunk` views per chunk on `lanes`
// streams over the items (every view, or `sample` evenly spaced views per
// scene when sample > 0); max_dups[b] is scene b's largest per-view pair
// count.  When the layout outgrows the memory it has, it synchronises the
// device and reallocates: never while a stream is capturing.
int drain_prepare(DrainLayout* d, const std::vector<scoup_batch_item>& items, const std::vector<int64_t>& max_dups,
                  int C, int K, int accum_mode, int chunk, int lanes, int sample);

// Enqueues the batch: set-up on `st`, chunks on the lane streams (forked from
// and joined back into `st`), Top-K on `st`; stats_dev (or null) receives a
// copy of each scene's header.  Capturable.
int drain_enqueue(DrainLayout* d, const std::vector<scoup_batch_item>& items, int C, int K, int accum_mode,
                  int warp_w, const cudaStream_t* lane_st, const cudaEvent_t* join_ev, cudaEvent_t fork_ev,
                  WsHeader* stats_dev, cudaStream_t st);

void drain_release(DrainLayout* d);

}  // namespace scoup
