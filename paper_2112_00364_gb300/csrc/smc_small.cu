// smc_small.cu -- a whole small run in one launch: every segment of a run whose
// tiles are warps (32 particles each), few enough for one CTA or one thread-block
// cluster, runs in one launch, with a CTA or cluster barrier as the checkpoint
// barrier of Algorithm 1 (Section 3.3's loop: propagate, combine, resample,
// repeat) instead of a kernel boundary per segment.
//
// Warp w of CTA r (its rank in the cluster; 0 without one) is tile
// r * (TPB / 32) + w of the run.  Each segment is the wave kernel's work with a
// barrier between the steps that need one:
//   combine   (k > 0) the previous segment's tile records (in this CTA's shared
//             memory, where every CTA of the cluster wrote its own: a load of 30
//             cycles instead of an L2 round trip) combined by each warp for
//             itself into exact integer offsets (smc_combine.cuh), the log-Z
//             increment, the resampling decision and the search scalars: the
//             same integers in every CTA, so the same decisions;
//   search    each particle's systematic-resampling ancestor (the running sums from
//             the shared memory of the ancestor's CTA) and the fused gather of its
//             state;
//   segment   blocks to the next checkpoint with per-warp PC-sorted dispatch;
//   epilogue  per warp: its power-of-two reference, integer weights, running
//             sums and tile record (a warp is a tile, so the tile reference is
//             the warp's).
// The segment ends at the cluster barrier (release / acquire at cluster scope:
// the records, running sums and states written before it by any CTA of the
// cluster are visible to every CTA after it); the double-buffered records,
// sums and states of segment k are not written again before the barrier that
// ends segment k + 1, which every CTA reaches only after its reads of them.  No CTA
// reads another's shared memory after the last barrier, so each may then end.  The
// first remote store comes after a cluster barrier at the start: every CTA is
// resident by then.
// The tiles, their rounding and the combine's integers are those of the wave
// kernel for the same N, so a run gives the same bits here, alone through the
// waves, batched and served.  The barriers are the hardware's (every CTA of a
// cluster is resident at once); nothing spins.
#include <cuda_runtime.h>

#include <mutex>

#include "smc_engine.h"
#include "smc_internal.h"
#include "smc_step.cuh"

namespace smc {

constexpr int kSmallMaxTiles = 32;

__device__ __forceinline__ unsigned cluster_rank() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}

// The cluster barrier in its two halves: the writes of every thread of the
// cluster before its arrive are visible to every thread after its wait; work
// between the two overlaps the other CTAs' arrival.
__device__ __forceinline__ void cluster_arrive() {
  asm volatile("barrier.cluster.arrive.release;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
  asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}

// A store to, and a load from, the shared memory of CTA `rank` of the cluster at
// the address that `p` has in this CTA's (without a cluster: this CTA's own).
__device__ __forceinline__ unsigned smem_at(const void* p, unsigned rank) {
  unsigned a = (unsigned)__cvta_generic_to_shared(p), r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
  return r;
}
__device__ __forceinline__ void store_to_cta(longlong2* p, longlong2 v, unsigned rank) {
  asm volatile("st.shared::cluster.v2.s64 [%0], {%1, %2};"
               :: "r"(smem_at(p, rank)), "l"(v.x), "l"(v.y) : "memory");
}
__device__ __forceinline__ void store_to_cta(long long* p, long long v, unsigned rank) {
  asm volatile("st.shared::cluster.s64 [%0], %1;" :: "r"(smem_at(p, rank)), "l"(v) : "memory");
}
__device__ __forceinline__ long long load_from_cta(const long long* p, unsigned rank) {
  long long v;
  asm volatile("ld.shared::cluster.s64 %0, [%1];" : "=l"(v) : "r"(smem_at(p, rank)) : "memory");
  return v;
}

// systematic_search for one warp of a small run (tiles of 32 particles): each
// lane's tile from the offsets as there; then, per distinct tile among the
// lanes (one or two, the offsets being non-decreasing), the tile's 32 running
// sums in one load (lane l holds E_{j0+l}, from the shared memory of the tile's CTA)
// and every lane of that tile finds
// its first j with E_j > F by a binary search over the shuffled values.  The
// same ancestors and near-boundary flags as systematic_search, which reads a tile's
// sums in two rounds; a tile here is one warp.  Every lane calls it;
// `want` marks the lanes whose offset is searched.
template <int WPC, bool CL>
__device__ __forceinline__ int small_search(int i, bool want, const RunDev& A, const SearchCtx& X,
                                            const long long (*E)[32], bool* near) {
  constexpr unsigned kAll = 0xffffffffu;
  const int N = A.N, T = A.n_tiles, lane = threadIdx.x & 31;
  int a = i, t = -1;
  bool nr = false, need = false;
  long long F = 0, tolF = 0, Z = 0;
  if (want) {
    const Q64 z = q_add(X.z0, q_mul_u32((unsigned)i, X.d));
    Z = (long long)z.hi;
    int lo = 0, hi = T;  // O_0 = 0 <= z
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (X.O[mid] <= Z)
        lo = mid;
      else
        hi = mid - 1;
    }
    if (lo >= T) {  // above the last offset (rounding at the top)
      nr = Z - X.O[T] < X.tolZ;
      a = N - 1;
    } else {
      t = lo;
      const int sh = X.kmax - X.ks[t] + X.G;
      F = q_threshold(z, X.O[t], sh);
      tolF = shl_sat(X.tolZ, sh);
      need = true;
    }
  }
  unsigned pending = __ballot_sync(kAll, need);
  while (pending) {
    const int tg = __shfl_sync(kAll, t, __ffs(pending) - 1);
    const int j0 = tg * 32, len = min(32, N - j0);
    long long e = 0x7FFFFFFFFFFFFFFFll;
    if (lane < len) e = CL ? load_from_cta(&E[tg % WPC][lane], (unsigned)(tg / WPC)) : E[tg][lane];
    // pos = #{ l < len : E_{j0+l} <= F } (the sums are non-decreasing)
    int pos = 0;
#pragma unroll
    for (int step = 16; step >= 1; step >>= 1) {
      const long long v = __shfl_sync(kAll, e, pos + step - 1);
      if (v <= F) pos += step;
    }
    const long long e31 = __shfl_sync(kAll, e, 31);
    if (pos == 31 && e31 <= F) pos = 32;
    pos = min(pos, len);
    const long long El = __shfl_sync(kAll, e, min(pos, 31));
    const long long Eb = __shfl_sync(kAll, e, max(pos - 1, 0));
    const bool mine = need && t == tg;
    if (mine) {
      nr = F - (pos > 0 ? Eb : 0ll) < tolF;
      if (pos < len) {
        a = j0 + pos;
        nr = nr || El - F <= tolF;
      } else if (j0 + len < N) {  // the first element of the next tile
        a = j0 + len;
        nr = nr || X.O[tg + 1] - Z <= X.tolZ;
      } else {
        a = N - 1;
      }
    }
    pending &= ~__ballot_sync(kAll, mine);
  }
  *near = nr;
  return a;
}

// The warp's sum of a 64-bit per-lane count, added by lane 0.
__device__ __forceinline__ void warp_add_u64_wide(unsigned long long* dst, unsigned long long v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0 && v) atomicAdd(dst, v);
}

// The warp's sum of a 32-bit value per lane, exactly, to every lane.
__device__ __forceinline__ unsigned long long warp_sum_u32(unsigned v) {
  const unsigned lo = __reduce_add_sync(0xffffffffu, v & 0xffffu);
  const unsigned hi = __reduce_add_sync(0xffffffffu, v >> 16);
  return lo + ((unsigned long long)hi << 16);
}

// The combine of at most 32 tiles by one warp, lane t holding tile t: the
// integers of combine_offsets (the same k_max, coarsening G, unit totals,
// exact offsets and S, and pieces of the sum of squared weights, so the same
// effective sample size) from warp shuffles, with no CTA barrier.  Writes
// O[0..nt] (O[nt] = S) and ks[0..nt) to the warp's own shared arrays.
__device__ __forceinline__ Combined combine_warp(const TileRec* rec, int nt, const long long* q,
                                                 long long* O, int* ks) {
  constexpr unsigned kAll = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  TileRec r;
  r.s = 0;
  r.k = kDeadTile;
  r.alive = 0;
  if (lane < nt) r = rec[lane];
  Combined c;
  c.kmax = __reduce_max_sync(kAll, r.k);
  c.alive = __any_sync(kAll, r.alive) ? 1 : 0;
  c.G = 0;
  c.S = 0;
  c.ess = 0.0;
  if (lane < nt) ks[lane] = r.k;
  if (c.kmax == kDeadTile) {
    __syncwarp();
    return c;
  }
  long long b = lane < nt ? magnitude(r.s, r.k, c.kmax) : 0;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) b += __shfl_xor_sync(kAll, b, o);
  c.G = (64 - __clzll(b)) + 20 - 62;
  const long long v = lane < nt ? to_run_units(r.s, r.k, c.kmax, c.G) : 0;
  long long inc = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const long long y = __shfl_up_sync(kAll, inc, o);
    if (lane >= o) inc += y;
  }
  c.S = __shfl_sync(kAll, inc, 31);
  if (lane < nt) O[lane] = inc - v;
  if (lane == 0) O[nt] = c.S;
  if (q) {
    unsigned long long f = 0, l = 0, h = 0;
    if (lane < nt && r.k != kDeadTile)
      add_squares((unsigned long long)q[lane], c.kmax - r.k, &f, &l, &h);
    c.ess = ess_of(warp_sum_u32((unsigned)f), warp_sum_u32((unsigned)l), warp_sum_u32((unsigned)h),
                   c.S, c.G);
  }
  __syncwarp();
  return c;
}

// CL: launched as one cluster of ceil(n_tiles / (TPB / 32)) CTAs (else one CTA),
// each with one warp more than its tiles: that of rank 0 closes the segments (log
// Z, its records), off every tile's path.
template <class M, int TPB, bool CL>
__global__ void __launch_bounds__(TPB + (CL ? 32 : 0), 1) small_run_kernel(const __grid_constant__ RunDev A) {
  using R = typename M::R;
  constexpr int WPC = TPB / 32;
  static_assert(CL || WPC >= 16, "one CTA holds the whole run");
  constexpr int NT = TPB + (CL ? 32 : 0);
  __shared__ long long sh_O[NT / 32][kSmallMaxTiles + 1];  // each warp's own offsets
  __shared__ int sh_ks[NT / 32][kSmallMaxTiles + 1];
  // double-buffered by segment parity: every tile's record (and sum of squared
  // weights), and the running sums of this CTA's tiles
  __shared__ __align__(16) TileRec sh_rec[2][kSmallMaxTiles];
  __shared__ long long sh_tq[2][kSmallMaxTiles];
  __shared__ long long sh_E[2][WPC][32];
  if (CL) {
    cluster_arrive();
    cluster_wait();
  }
  RunState* rs = A.rs;
  const int N = A.N;
  const int wid = (int)(threadIdx.x >> 5);
  const bool extra = CL && wid == WPC;  // the warp without a tile
  // the thread that closes each segment
  const bool closes = CL ? extra && cluster_rank() == 0 && (threadIdx.x & 31) == 0 : threadIdx.x == 0;
  const int t = (CL ? (int)cluster_rank() * WPC : 0) + wid;
  const int lane = threadIdx.x & 31;
  const int i = t * 32 + lane;  // the tile of this path is 32 particles
  const int ctas = (int)gridDim.x;  // (the cluster is the grid)
  const bool tile_live = !extra && t < A.n_tiles;
  const bool valid = tile_live && i < N;
  // segment k - 1's closing (log Z, its records) waits for the barrier that
  // ends segment k, where it overlaps the other CTAs' arrival
  Combined c_close;
  bool resample_close = false;
  unsigned long long uf = 0;  // the uniform of the next search, drawn in the barrier's shadow
  // the run's counters, summed per lane over the segments and added once
  unsigned long long n_near = 0, n_overflow = 0, n_limit = 0, n_draws = 0, n_blocks = 0;
  typename M::Lane Ln;  // (what predraw() fills, for the next segment)
  for (int k = 0;; ++k) {
    const int nb = k & 1, cb = nb ^ 1;
    const StateView Sc = A.state[cb];
    const StateView Sn = A.state[nb];
    typename M::Lane L;
    Stream s{A.k0, A.k1, (uint32_t)i, (uint32_t)k, 0u, 0u, A.md.tab};
    if constexpr (M::PREDRAW) {
      L.z = Ln.z;
      L.drawn = k > 0;
      s.d = k > 0 ? 1 : 0;
    }
    bool near = false;
    if (k > 0) {
      const Combined c = combine_warp(sh_rec[cb], A.n_tiles, A.ess ? sh_tq[cb] : nullptr,
                                      sh_O[wid], sh_ks[wid]);
      const bool go_on = c.kmax != kDeadTile && c.alive && k < A.max_segments;
      const bool resample = decide_resample(A, c);
      if (!go_on) {  // the same c in every thread: a uniform exit
        if (closes) finish_segment(A, k, c, resample);
        break;
      }
      c_close = c;
      resample_close = resample;
      // the run's search scalars by each warp's lane 0, broadcast to its lanes
      unsigned long long q5[5] = {0ull, 0ull, 0ull, 0ull, 0ull};
      if (resample && lane == 0) {
        Q64 d, z0;
        long long tolZ;
        search_scalars(c, N, A.recip_n, uf, &d, &z0, &tolZ);
        q5[0] = d.hi;
        q5[1] = d.lo;
        q5[2] = z0.hi;
        q5[3] = z0.lo;
        q5[4] = (unsigned long long)tolZ;
      }
#pragma unroll
      for (int q = 0; q < 5; ++q) q5[q] = __shfl_sync(0xffffffffu, q5[q], 0);
      SearchCtx X;
      X.rec = nullptr;
      X.O = sh_O[wid];
      X.ks = sh_ks[wid];
      X.kmax = c.kmax;
      X.G = c.G;
      X.d = Q64{q5[0], q5[1]};
      X.z0 = Q64{q5[2], q5[3]};
      X.tolZ = (long long)q5[4];
      const int a_s = resample ? small_search<WPC, CL>(i, valid, A, X, sh_E[cb], &near) : i;
      if (valid) {
        const int row = A.record_all ? k - 1 : 0;
        int a = a_s;
        bool bad = false;
        if (SMC_DEBUG_CHECKS) {
          if (!(a >= 0 && a < N)) {
            debug_record(rs, 1, i);
            a = i;
            bad = true;
          }
          if (M::HAS_STACK) {
            const int spa = Sc.inf_(1, a, N);
            if (!(spa >= 0 && spa <= A.md.lam_stack_cap)) {
              debug_record(rs, 3, i);
              bad = true;
            }
          }
        }
        if (row < A.anc_rows) A.anc[(size_t)row * N + i] = a;
        if (bad) {
          M::init(L);
          L.pc = PC_STOP;
          L.logw = neg_inf<R>();
        } else if (resample) {
          M::gather(L, Sc, Sn, a, i, N, A.md);
        } else {
          M::gather(L, Sc, Sn, i, i, N, A.md);
          L.logw = (R)A.logw[i];
        }
      }
      n_near += near ? 1ull : 0ull;
    } else if (valid) {
      M::init(L);
    }
    if (SMC_DEBUG_CHECKS && valid && !(L.pc == PC_STOP || (L.pc >= 0 && L.pc < M::NB))) {
      debug_record(rs, 2, i);
      L.pc = PC_STOP;
      L.logw = neg_inf<R>();
    }
    const bool active = valid && L.pc != PC_STOP;
    const int n_exec = run_segment<M>(L, s, A.md, Sn, i, k, N, active);
    double lw = -INFINITY;
    int alive = 0;
    if (valid) {
      M::store(L, Sn, i, N);
      lw = widen(L.logw);
      A.logw[i] = lw;
      alive = L.pc != PC_STOP;
    }
    n_overflow += active ? (unsigned long long)L.overflow : 0ull;
    n_limit += active ? (unsigned long long)L.limited : 0ull;
    n_draws += valid ? (unsigned long long)s.d : 0ull;
    n_blocks += (unsigned long long)n_exec;
    // the tile's weights: a warp is a tile, so its reference is the warp's
    long long ef = 0;
    const double Mw = warp_max_key(lw);
    const int kt = is_neg_inf(Mw) ? kDeadTile : tile_exponent_fast(Mw);
    if (valid && kt != kDeadTile) {
      if (kt > -2048 && kt < 2048) {
        ef = weight_fix54(lw, kt, ref_q58_lo(kt), A.md.tab);
      } else {
        const double kd = (double)kt;
        const double dd = fma(-kd, kLn2Lo, fma(-kd, kLn2Hi, lw));
        ef = exp_fix54(dd, A.md.tab);
      }
    }
    const long long E = block_incl_scan_i64<32>(ef, nullptr);  // a warp scan
    if (tile_live) sh_E[nb][wid][lane] = E;
    if (A.ess) {
      const unsigned long long u = (unsigned long long)ef;
      const long long sq = (long long)((__umul64hi(u, u) << 10) | ((u * u) >> 54));
      const long long Q = __shfl_sync(0xffffffffu, block_incl_scan_i64<32>(sq, nullptr), 31);
      if (CL) {
        if (tile_live && lane < ctas) store_to_cta(&sh_tq[nb][t], Q, (unsigned)lane);
      } else if (tile_live && lane == 0) {
        sh_tq[nb][t] = Q;
      }
    }
    const int tile_alive = __any_sync(0xffffffffu, alive) ? 1 : 0;
    // the record to every CTA of the cluster, a lane each
    longlong2 rec;
    rec.x = __shfl_sync(0xffffffffu, E, 31);
    rec.y = (long long)(unsigned)kt | ((long long)tile_alive << 32);
    if (CL) {
      if (tile_live && lane < ctas) store_to_cta(reinterpret_cast<longlong2*>(&sh_rec[nb][t]), rec, (unsigned)lane);
    } else if (tile_live && lane == 0) {
      *reinterpret_cast<longlong2*>(&sh_rec[nb][t]) = rec;
    }
    // the segment's records, running sums and states, for the next combine
    if (CL) cluster_arrive();
    if (k > 0 && closes) finish_segment(A, k, c_close, resample_close);
    if constexpr (M::PREDRAW) {
      if (valid) {
        Stream sn{A.k0, A.k1, (uint32_t)i, (uint32_t)(k + 1), 0u, 0u, A.md.tab};
        M::predraw(Ln, sn);
      }
    }
    if (lane == 0) uf = search_uniform(A, k);
    if (CL)
      cluster_wait();
    else
      __syncthreads();
  }
  warp_add_u64_wide(&rs->n_near, n_near);
  warp_add_u64_wide(&rs->n_overflow, n_overflow);
  warp_add_u64_wide(&rs->n_limit, n_limit);
  warp_add_u64_wide(&rs->n_draws, n_draws);
  warp_add_u64_wide(&rs->n_blocks, n_blocks);
}

// One CTA: register-light models run up to 32 tiles (1024 threads, 64
// registers a thread); the tree and SEIR models up to 16 (512 threads).
// Cluster: up to 32 tiles for every model, 2 warps a CTA in clusters of up to
// 16 CTAs where the GPU schedules them, else 4 warps a CTA in up to 8.
int small_run_max_tiles(int kind, int launch_mode) {
  if (launch_mode == SMC_LAUNCH_CLUSTER) return kSmallMaxTiles;
  switch (kind) {
    case SMC_MODEL_LG:
    case SMC_MODEL_GEOMETRIC: return 32;
    default: return 16;
  }
}

namespace {
template <class M, int TPB>
cudaError_t launch_cluster(const RunDev& run, int n_tiles, cudaStream_t st) {
  auto kern = small_run_kernel<M, TPB, true>;
  static std::once_flag once;
  static cudaError_t attr = cudaSuccess;
  std::call_once(once, [&] {
    if (TPB / 32 * 8 < kSmallMaxTiles)
      attr = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  });
  if (attr != cudaSuccess) return attr;
  const unsigned ctas = (unsigned)((n_tiles + TPB / 32 - 1) / (TPB / 32));
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(ctas, 1, 1);
  cfg.blockDim = dim3(TPB + 32, 1, 1);
  cfg.dynamicSmemBytes = 0;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = ctas;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, run);
}

// Whether the GPU schedules clusters of 16 CTAs of 64 threads (asked once per
// process, for the device current at the first call).
bool wide_clusters() {
  static std::once_flag once;
  static bool wide = false;
  std::call_once(once, [] {
    auto kern = small_run_kernel<LgModel<double>, 64, true>;
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) {
      cudaGetLastError();
      return;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(16, 1, 1);
    cfg.blockDim = dim3(96, 1, 1);
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 16;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess) {
      cudaGetLastError();
      return;
    }
    wide = n > 0;
  });
  return wide;
}

template <class M>
cudaError_t launch_small_m(int launch_mode, int one_cta_tpb, const RunDev& run, int n_tiles,
                           cudaStream_t st) {
  if (launch_mode == SMC_LAUNCH_CLUSTER)
    return wide_clusters() ? launch_cluster<M, 64>(run, n_tiles, st)
                           : launch_cluster<M, 128>(run, n_tiles, st);
  if (one_cta_tpb == 1024)
    small_run_kernel<M, 1024, false><<<1, 1024, 0, st>>>(run);
  else
    small_run_kernel<M, 512, false><<<1, 512, 0, st>>>(run);
  return cudaGetLastError();
}

template <typename R>
cudaError_t launch_small_r(int kind, int launch_mode, const RunDev& run, int n_tiles,
                           cudaStream_t st) {
  switch (kind) {
    case SMC_MODEL_LG: return launch_small_m<LgModel<R>>(launch_mode, 1024, run, n_tiles, st);
    case SMC_MODEL_GEOMETRIC: return launch_small_m<GeoModel<R>>(launch_mode, 1024, run, n_tiles, st);
    case SMC_MODEL_SEIR: return launch_small_m<SeirModel<R>>(launch_mode, 512, run, n_tiles, st);
    case SMC_MODEL_CRBD:
      return launch_small_m<TreeModel<R, false>>(launch_mode, 512, run, n_tiles, st);
    case SMC_MODEL_RATESHIFT:
      return launch_small_m<TreeModel<R, true>>(launch_mode, 512, run, n_tiles, st);
    default: return launch_small_m<TreeDsModel<R>>(launch_mode, 512, run, n_tiles, st);
  }
}
}  // namespace

cudaError_t launch_small_run(int kind, int precision, int launch_mode, const RunDev& run,
                             int n_tiles, cudaStream_t st) {
  return precision == SMC_PREC_FP32 ? launch_small_r<float>(kind, launch_mode, run, n_tiles, st)
                                    : launch_small_r<double>(kind, launch_mode, run, n_tiles, st);
}

}  // namespace smc
