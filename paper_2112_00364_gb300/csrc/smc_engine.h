// smc_engine.h -- structures shared by the run, batch and server paths.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>
#include <utility>
#include <vector>

#include "../../include/smc.h"
#include "smc_combine.cuh"
#include "smc_models.cuh"

namespace smc {

constexpr int kMaxAncRows = 4096;
constexpr int kMaxSegments = 1 << 24;
constexpr int kUnboundedSegments = 1 << 20;
constexpr int64_t kMaxParticles = (int64_t)0x7fffffff - 256;

// Per-run device state (one struct per run, in the run's workspace).
struct RunState {
  double log_z, m, S;
  double log_z_closed;  // log Z without a closure made only because the step limit ended the run
  // the next search's scalars when the run combines in one CTA: S / N and
  // u S / N in 64.64 fixed point, and the boundary tolerance (units U)
  unsigned long long d_hi, d_lo, z0_hi, z0_lo;
  long long tolZ;
  unsigned long long n_near, n_overflow, n_limit;
  unsigned long long n_draws, n_blocks;  // Philox blocks drawn by the model, blocks executed
  int32_t done, status, n_segments, n_resamples;
  uint32_t arrive;
  int32_t kmax, G;        // the run's reference exponent and coarsening (one-CTA combine)
  int32_t resample;       // the one-CTA combine's decision for the next wave
  int32_t n_ess_near;     // ESS decisions within 1e-9 of the threshold
  // checking build (SMC_DEBUG_CHECKS): the first out-of-range access found and
  // skipped (code: 1 ancestor, 2 block index, 3 stack pointer, 4 dispatch), its
  // particle, and how many were found
  int32_t dbg_code, dbg_pad;
  long long dbg_index;
  unsigned long long dbg_count;
};

// Everything a CTA needs about its run (copied to shared memory per CTA).
struct RunDev {
  ModelDev md;
  StateView state[2];
  double* logw;       // [N] log-weights of the latest segment (f64; FP32 values widened)
  // [n_tiles][pad] running sums of the weights x 2^54 (int64) within each warp of a tile
  // (pad: the tile in whole warps), double-buffered by segment parity, and, for
  // tiles of more than one warp, [n_tiles][8] the warps' ends in the tile's running sum
  long long* E[2];
  long long* ends[2];
  TileRec* rec[2];    // [n_tiles] tile reductions, double-buffered by segment parity
  long long* tq[2];   // [n_tiles] ESS mode: the tiles' sums of squared weights (units 2^-54 of 2^(2 k_t))
  int32_t* dec;       // [max_segments] 1 where the population was resampled after checkpoint k
  long long* tile_O;  // [n_tiles + 1] offsets in the run's unit, O_T = S (runs combined in one CTA)
  int32_t* anc;       // ancestor rows
  double* incr;       // [max_segments] per-segment log-Z increments
  RunState* rs;
  double log_n;                // log N, computed on the host
  unsigned long long recip_n;  // floor((2^64 - 1) / N), the search scalars' divisor
  double ess_tau;       // 0: resample after every checkpoint; > 0: only when ESS < ess_tau N
  double ess_target;    // ess_tau N
  int N, n_tiles, tile, pad, max_segments, record_all, anc_rows;
  unsigned start_wave;  // wave index of the run's segment 0 (segment k runs in wave start_wave + k)
  int redundant;        // combine a segment's tiles in every CTA of the next wave (else in the last CTA)
  int ess;              // ess_tau > 0 (an integer flag for the kernel's branches)
  uint32_t k0, k1;
  // resume from a snapshot: segment resume_k - 1 loads the population (device copies)
  int resume_k;
  const double* snap_logw;
  const double* snap_real;
  const int32_t* snap_int;
  const double* snap_stack;
};

// A run's outputs for the collecting kernel: sources in the run's workspace, and
// destinations in device memory (NULL: not wanted).
struct CollectJob {
  StateView state[2];
  const double* src_logw;
  const int32_t* src_anc;
  const int32_t* dec;
  const RunState* rs;
  double *log_z, *logw, *real, *stack;
  int32_t *ints, *anc, *resampled;
  int N, n_real, n_int, cap, fp32, record_all, anc_rows, res_rows, max_segments;
  int parts;  // a batch's job: its CTAs
};
static_assert(sizeof(CollectJob) % 8 == 0, "the CTA map follows the jobs");

struct Layout {
  size_t real[2], ints[2], stack[2], logw, E[2], ends[2], rec[2], tq[2], dec, tO, rs, anc, incr,
      fin_real, fin_int, fin_stack, stage, snap, total;
  int n_tiles, tile, pad, anc_rows, max_segments;
};

// One model and CTA size among the runs of a set: a wave of the set is one launch
// per chain, and a chain's launches depend on one another only (every run belongs
// to one chain).
struct WaveChain {
  int kind = 0, bucket = 0, n_ctas = 0;
  const int2* map = nullptr;  // CTA -> (run, tile)
  // The runs of a set that starts together lie in the map from the longest to the
  // shortest, so the CTAs of those that wave w still advances are its first ones:
  // {waves, CTAs up to this run} with ascending CTAs, descending waves.  A wave
  // launches those alone: the CTAs of finished runs only read their run's state and
  // return, but of a batch of 512 uneven runs 70% were such (132 -> 115 ms without
  // them).  Empty: every CTA every wave (a server's runs start at different waves).
  std::vector<std::pair<int, int>> live;
  int ctas_at(unsigned wave) const {
    if (live.empty()) return n_ctas;
    int lo = 0, hi = (int)live.size();  // the runs with waves > wave
    while (lo < hi) {
      const int mid = (lo + hi) / 2;
      if ((unsigned)live[mid].first > wave) lo = mid + 1;
      else hi = mid;
    }
    return lo > 0 ? live[lo - 1].second : 0;
  }
  bool operator==(const WaveChain& o) const {
    return kind == o.kind && bucket == o.bucket && n_ctas == o.n_ctas && map == o.map &&
           live == o.live;
  }
};
constexpr int kMaxChains = 6 * 4;
constexpr int kChainStreams = 8;  // two models in four CTA sizes have a stream each

// Device addresses of one set's run table and its chains.
struct WavePlan {
  const RunDev* runs = nullptr;
  std::vector<WaveChain> chains;
};

// Streams for a set's chains beside the stream its caller works on, so that a
// chain's waves need not wait for the slowest CTAs of the others' (on one stream
// every launch waits for the launch before it).  fork(): the chains' work waits for
// what `main` holds so far; join(): `main` waits for the chains' work so far.
// Chain i runs on stream i modulo the number of streams.  Used by one batch call
// or one server at a time; its streams are idle when it is destroyed (after a join
// that the owner has waited for).
class ChainStreams {
 public:
  ChainStreams() = default;
  ChainStreams(const ChainStreams&) = delete;
  ChainStreams& operator=(const ChainStreams&) = delete;
  ~ChainStreams();
  cudaError_t init(int n);  // at least n streams
  cudaError_t fork(cudaStream_t main, int chains);
  cudaError_t join(cudaStream_t main, int chains);
  cudaStream_t at(int chain) const { return s_[(size_t)chain % s_.size()]; }
  int size() const { return (int)s_.size(); }

 private:
  std::vector<cudaStream_t> s_;
  std::vector<cudaEvent_t> done_;
  cudaEvent_t ready_ = nullptr;
};

// The streams of one batch call: a set that an earlier call left idle, or a new one; left
// for later calls once idle() was called, destroyed otherwise (after an error).
class BorrowedStreams {
 public:
  BorrowedStreams() = default;
  BorrowedStreams(const BorrowedStreams&) = delete;
  BorrowedStreams& operator=(const BorrowedStreams&) = delete;
  ~BorrowedStreams();
  cudaError_t take(int n);
  void idle() { idle_ = true; }
  ChainStreams* get() const { return set_; }

 private:
  ChainStreams* set_ = nullptr;
  int dev_ = 0;
  bool idle_ = false;
};

// An instantiated CUDA graph of a known-length sequence of waves and the wave
// plan it was captured for.
struct GraphCache {
  cudaGraphExec_t exec = nullptr;
  WavePlan plan;
  int precision = -1, waves = 0, launches = 0;
};
void graph_cache_clear(GraphCache* g);

// Device blocks through a small cache of blocks freed by destroyed model
// handles (smc_engine.cu): *got receives the block's size (at least bytes).
cudaError_t block_alloc(void** p, size_t* got, size_t bytes);
void block_free(void* p, size_t bytes, int dev);

// A whole run in one launch (smc_small.cu): for runs of 32-particle tiles, at
// most small_run_max_tiles(kind, launch_mode) of them; launch_mode
// SMC_LAUNCH_ONE_CTA (grid 1) or SMC_LAUNCH_CLUSTER (one thread-block cluster).
int small_run_max_tiles(int kind, int launch_mode);
cudaError_t launch_small_run(int kind, int precision, int launch_mode, const RunDev& run,
                             int n_tiles, cudaStream_t st);

}  // namespace smc

struct smc_model_s {
  smc_model_desc desc;
  smc::ModelDev md;
  int32_t n_real, n_int, stack_cap, n_segments_known;
  int32_t n_real_state;  // real fields kept in PSTATE (>= n_real; extra ones are internal)
  int dev = 0;                // the device the handle's memory is on
  void* dev_blob = nullptr;  // observations / tree arrays
  size_t blob_bytes = 0;
  void* ws = nullptr;        // cached workspace of smc_run
  size_t ws_bytes = 0;
  cudaEvent_t ev0 = nullptr, ev1 = nullptr;
  std::vector<cudaEvent_t> ev_seg;  // per-launch timing pairs (time_kernels)
  std::vector<char> staging;        // host staging of the run table
  char* pin = nullptr;              // smc_run's pinned copy of it (uploaded without a wait)
  size_t pin_bytes = 0;
  cudaEvent_t pin_ev = nullptr;     // recorded after that upload: the buffer is free again
  char* pin_out = nullptr;          // smc_run's pinned copy of the run's state and small host results
  size_t pin_out_bytes = 0;
  smc::GraphCache graph;            // smc_run's captured waves (SMC_LAUNCH_GRAPH)
};

namespace smc {

int model_fields(int kind, int* n_real, int* n_int);
// This device's log / exp tables (filled on first use per device).
smc_status math_table(const MathTab** out);
int tile_for(int64_t N);
int bucket_for(int tile);
// The combine placement of a run (the same results either way): in every CTA
// of the next wave when latency matters (`single`: a run alone, up to
// redundant_cap tiles), else only for runs of at most 32 tiles.
int combine_in_every_cta(int tile, int n_tiles, bool single);
Layout make_layout(const smc_model_s* m, const smc_run_cfg* c);
RunDev make_rundev(const smc_model_s* m, const smc_run_cfg* c, const Layout& Ly, char* ws);
size_t wave_meta_bytes(const std::vector<RunDev>& runs);
smc_status upload_wave(const std::vector<RunDev>& runs, void* meta, cudaStream_t st, WavePlan* W,
                       std::vector<char>* staging, char* pinned = nullptr,
                       const std::vector<int>* waves = nullptr);
// The run table and CTA maps of a set of runs into `host` (at least
// wave_meta_bytes(runs)), the plan for them at the device address `dev`; returns
// the bytes to copy.  `waves`: how many waves, from wave 0, each run takes at most.
size_t fill_plan(const std::vector<RunDev>& runs, char* host, void* dev, WavePlan* W,
                 const std::vector<int>* waves = nullptr);
// One wave: every chain's launch, on `st`, or each on its own stream with `streams`;
// adds the number of launches to *launched.
cudaError_t launch_wave(const WavePlan& W, int precision, cudaStream_t st, unsigned wave,
                        const ChainStreams* streams = nullptr, int* launched = nullptr);
// (alone: no other chain runs beside this one; dense: the wave's CTAs do not all fit at
// once, resident_threads())
template <int KIND, typename R>
cudaError_t launch_kind(const WaveChain& c, int n_ctas, const RunDev* runs, cudaStream_t st,
                        unsigned wave, bool alone, bool dense);
smc_status collect_run(const smc_model_s* m, const smc_run_cfg* c, const Layout& Ly, char* ws,
                       const RunDev& A, const RunState& hrs, smc_result* r, cudaStream_t cs);
smc_status check_cfg(const smc_model_s* m, const smc_run_cfg* c);
smc_status check_result(const smc_result* r);

}  // namespace smc
