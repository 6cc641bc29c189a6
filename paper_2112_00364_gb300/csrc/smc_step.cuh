// smc_step.cuh -- one tile of one run for one segment: the body of every
// segment kernel (wave_kernel below and the one-launch kernels of smc_small.cu).  Algorithm 1 in the RootPPL loop order of Section 3.3: the
// previous segment's tiles combined into exact integer offsets, the log-Z
// increment and the resampling decision; the systematic search and the
// particle duplication fused into the load; blocks run to the next checkpoint;
// the tile's weights, running sums and record.
#pragma once
#include <cuda_runtime.h>

#include "smc_combine.cuh"
#include "smc_device.cuh"
#include "smc_engine.h"
#include "smc_models.cuh"

#ifndef SMC_DEBUG_CHECKS
#define SMC_DEBUG_CHECKS 0
#endif

namespace smc {

// Checking build: record an out-of-range access (the caller skips it).
__device__ __forceinline__ void debug_record(RunState* rs, int code, long long index) {
  atomicAdd(&rs->dbg_count, 1ull);
  if (atomicCAS(&rs->dbg_code, 0, code) == 0) rs->dbg_index = index;
}

__device__ __forceinline__ void warp_add_u64(unsigned long long* dst, unsigned long long v) {
  v = __reduce_add_sync(0xffffffffu, (unsigned)v);
  if ((threadIdx.x & 31) == 0 && v) atomicAdd(dst, v);
}

// Whether to resample after checkpoint k-1 (the same in every CTA: c is).
__device__ __forceinline__ bool decide_resample(const RunDev& A, const Combined& c) {
  return !A.ess || c.ess < A.ess_target;
}

// Finish segment k-1 of the run from its combined offsets (one thread):
// log Z += k_max ln 2 + (log S - log N) with S = S_units U, the increment
// record, and the end of the run.  Returns whether segment k runs.
__device__ __forceinline__ bool finish_segment(const RunDev& A, int k, const Combined& c,
                                               bool resample) {
  RunState* rs = A.rs;
  if (c.kmax == kDeadTile) {
    rs->log_z = -INFINITY;
    rs->log_z_closed = -INFINITY;
    rs->m = -INFINITY;
    rs->S = 0.0;
    A.incr[k - 1] = -INFINITY;
    rs->status = SMC_EDEGENERATE;
    rs->done = 1;
    rs->n_segments = k;
    return false;
  }
  const double Sd = (double)c.S;
  const double inc = (double)(c.kmax - 54 + c.G) * kLn2 + (tang_log(Sd, A.md.tab) - A.log_n);
  const bool go_on = c.alive && k < A.max_segments;
  // the accumulated weights are closed into log Z when the population is
  // resampled, at the end and at the step limit
  const bool close = !go_on || resample;
  if (close) rs->log_z = rs->log_z + inc;
  if (!(c.alive && k >= A.max_segments)) rs->log_z_closed = rs->log_z;  // not a step-limit closure
  A.incr[k - 1] = close ? inc : 0.0;
  rs->m = (double)c.kmax * kLn2;
  rs->S = Sd * pow2i(c.G - 54);
  rs->n_segments = k;
  if (go_on) {
    A.dec[k - 1] = resample ? 1 : 0;
    rs->n_resamples += resample ? 1 : 0;
    if (A.ess && fabs(c.ess - A.ess_target) <= 1e-9 * A.ess_target) rs->n_ess_near += 1;
  }
  if (!c.alive) {
    rs->done = 1;
  } else if (!go_on) {
    rs->status = SMC_ESTEPLIMIT;
    rs->done = 1;
  }
  return go_on;
}

// u 2^64 of the uniform of the search after checkpoint k.
__device__ __forceinline__ unsigned long long search_uniform(const RunDev& A, int k) {
  return frac64(Unif<double>::first(philox(0u, (uint32_t)k, 0u, 1u, A.k0, A.k1)));
}

// What the search of segment k needs about segment k-1's weights.
struct SearchCtx {
  const long long* O;  // offsets in units U, O[T] = S
  const int* ks;       // tile reference exponents (shared memory), or NULL: read the records
  const TileRec* rec;
  int kmax, G;
  Q64 d, z0;           // S / N and u S / N in 64.64 (units U)
  long long tolZ;      // 1e-12 N on the q scale, in units U
};

// The run's search scalars from its combined total (one thread); uf = u 2^64.
__device__ __forceinline__ void search_scalars(const Combined& c, int N, unsigned long long recip_n,
                                               unsigned long long uf, Q64* d, Q64* z0,
                                               long long* tolZ) {
  *d = q_ratio((unsigned long long)c.S, (unsigned long long)N, recip_n);
  *z0 = q_scale(uf, *d);
  *tolZ = floor_i64(kBoundaryEps * (double)c.S);
}

// The tile of an offset: t = max{ t : O_t <= Z } in [0, T], and O_t.  Every lane
// of the warp calls it; the lanes' Z are non-decreasing.  The warp's 32
// consecutive offsets span few tiles, so one window of 32 tile offsets, one
// load a lane, holds them all: around the CTA's own tile when the offsets are in
// global memory (systematic ancestors lie near their particle: the window holds
// them but for a population whose weights are very uneven across its tiles), by
// one 32-way step through shared memory when they are there; a 32-way descent
// finds the window otherwise.  One or two rounds of loads against the log2 T
// dependent ones of a binary search per lane (12 L2 round trips at 4,096 tiles).
// kShared: O is in shared memory and T < 1024.
__device__ __forceinline__ int find_tile(long long Z, const long long* O, int T, bool shared_O,
                                         int near_t, long long* Ot) {
  constexpr unsigned kAll = 0xffffffffu;
  constexpr long long kTop = 0x7FFFFFFFFFFFFFFFll;
  const int lane = threadIdx.x & 31;
  const long long Zf = __shfl_sync(kAll, Z, 0);
  const long long Zl = __shfl_sync(kAll, Z, 31);
  int w0 = shared_O ? 0 : max(0, min(near_t - 15, T - 31));
  long long val = kTop;
  bool have = false;
  if (!shared_O) {
    if (w0 + lane <= T) val = O[w0 + lane];
    const unsigned le = __ballot_sync(kAll, val <= Zf);
    have = le != 0u && le != kAll;
  }
  if (!have) {  // 32-way descent to the window that holds the first lane's tile
    int span = T + 1;
    w0 = 0;
    while (span > 32) {
      const int step = (span + 31) >> 5, at = lane * step;
      const long long v = at < span ? O[w0 + at] : kTop;
      const int s = __popc(__ballot_sync(kAll, v <= Zf)) - 1;  // O_w0 <= Zf
      w0 += s * step;
      span = min(step, span - s * step);
    }
    val = w0 + lane <= T ? O[w0 + lane] : kTop;
  }
  const int cf = __popc(__ballot_sync(kAll, val <= Zf)) - 1;
  const int cl = __popc(__ballot_sync(kAll, val <= Zl)) - 1;
  int p = cf;
  if (cl != cf) {  // the lanes lie in different tiles
    p = 0;
#pragma unroll
    for (int step = 16; step >= 1; step >>= 1) {
      const long long v = __shfl_sync(kAll, val, p + step);
      if (v <= Z) p += step;
    }
  }
  *Ot = __shfl_sync(kAll, val, p);
  int t = w0 + p;
  if (cl == 31 && p == 31 && t < T) {  // beyond the window: a binary search
    int hi = T;
    while (t < hi) {
      const int mid = (t + hi + 1) >> 1;
      if (O[mid] <= Z)
        t = mid;
      else
        hi = mid - 1;
    }
    *Ot = O[t];
  }
  return t;
}

// a_i = min{ j : q_j > y } for y = i + u, with q_j = P_j N / S and P_j the
// running sum of the weights; on the P scale in units U the offset is
// z_i = z_0 + i S / N (64.64 fixed point, exact and non-decreasing in i).  The
// tile is t = max{ t : O_t <= z } (N - 1 if z lies above every offset); inside
// it P_j = O_t + E_j 2^-(k_max - k_t + G), so P_j > z <=> E_j > floor((z - O_t)
// 2^(k_max - k_t + G)) (E_j is an integer): one threshold F per particle.  The
// tile's running sums are kept as its warps' own (E_j = C_{c-1} + e_j for warp c of
// the tile) with the warps' ends C_c in one 64-byte row a tile, so the search is
// the row (which warp: the first C_c > F), eight of the warp's 32 sums and the
// four between two of those: two rounds of loads, the third from lines the second
// brought.  Bound: the latency of those rounds and issue; with a binary search per
// lane over the tiles and an 8-ary search over a whole tile's sums (12 + 3 rounds
// at 4,096 tiles) a wave of 2^20 particles took 105 us instead of 77 with the
// linear-Gaussian model, 158 instead of 144 with the rate-shift model.  If no
// element of tile t qualifies, the first element of tile t+1 does.  The offset is
// flagged when it lies within 1e-12 N of q_a or q_{a-1}, measured in the same
// units.  Integer arithmetic only.  Every lane of the warp calls it (i of the
// lanes past the last particle repeats that particle).
__device__ __forceinline__ int systematic_search(int i, int near_t, const RunDev& A,
                                                 const SearchCtx& X,
                                                 const long long* __restrict__ E,
                                                 const long long* __restrict__ ends, bool* near) {
  const int N = A.N, T = A.n_tiles;
  const Q64 z = q_add(X.z0, q_mul_u32((unsigned)i, X.d));
  const long long Z = (long long)z.hi;
  long long Ot;
  const int t = find_tile(Z, X.O, T, X.ks != nullptr, near_t, &Ot);
  if (t >= T) {  // above the last offset (rounding at the top)
    *near = Z - Ot < X.tolZ;
    return N - 1;
  }
  const int kt = X.ks ? X.ks[t] : __ldcg(&X.rec[t].k);
  const int pad = A.pad;
  long long base = 0;  // the sum before the warp's first element
  int c = 0;
  long long C[8];
  if (pad > 32) {
    const longlong2* p = reinterpret_cast<const longlong2*>(ends + (size_t)t * 8);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const longlong2 v = p[q];
      C[2 * q] = v.x;
      C[2 * q + 1] = v.y;
    }
  }
  const int sh = X.kmax - kt + X.G;
  const long long F = q_threshold(z, Ot, sh);
  const long long tolF = shl_sat(X.tolZ, sh);
  if (pad > 32) {
#pragma unroll
    for (int q = 0; q < 8; ++q)
      if (C[q] <= F) {
        base = C[q];
        c = q + 1;
      }
  }
  const int j0 = t * A.tile, j1 = min(N, j0 + A.tile);
  int a = -1;
  long long Eb = base;  // E_{a-1}, or the tile's total when no element qualifies
  long long El = 0;
  if (c < 8) {
    const long long* e = E + ((size_t)t * pad + (size_t)c * 32);
    const long long f = F - base;
    long long v[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) v[q] = e[4 * q + 3];
    int m = 0;
    long long b = 0;
#pragma unroll
    for (int q = 0; q < 8; ++q)
      if (v[q] <= f) {
        b = v[q];
        m = q + 1;
      }
    if (m < 8) {
      const longlong2* p = reinterpret_cast<const longlong2*>(e + 4 * m);
      const longlong2 v0 = p[0], v1 = p[1];
      int l = 4 * m;
      El = v0.x;
      if (v0.x <= f) {
        b = v0.x;
        El = v0.y;
        l += 1;
        if (v0.y <= f) {
          b = v0.y;
          El = v1.x;
          l += 1;
          if (v1.x <= f) {
            b = v1.x;
            El = v1.y;
            l += 1;
          }
        }
      }
      a = j0 + c * 32 + l;
      El += base;
    }
    Eb += b;
  }
  bool nr = F - Eb < tolF;
  if (a >= 0) {
    nr = nr || El - F <= tolF;
  } else if (j1 < N) {  // the first element of the next tile
    a = j1;
    nr = nr || X.O[t + 1] - Z <= X.tolZ;
  } else {
    a = N - 1;
  }
  *near = nr;
  return a;
}

// A CTA's shared memory.
template <int TPB>
struct StepShared {
  double red[combine_scratch(TPB)];  // combine_offsets' reductions
  double ess;                      // its effective sample size
  unsigned long long scal[5];      // the search scalars
  unsigned long long uf;           // u 2^64 of the search they are for
  long long sum[TPB / 32], sq[TPB / 32];  // the warps' weight sums (and of their squares)
  unsigned draws[TPB / 32], execs[TPB / 32];
  int kw[TPB / 32], last, resample;
  long long O[redundant_cap(TPB)];  // the offsets of a run combined in every CTA
  int ks[redundant_cap(TPB)];       // and its tiles' reference exponents
};

// What the combine's threads publish: for a run combined in every CTA, the
// decision and the search scalars in shared memory, a thread each.
template <int TPB>
struct PublishShared {
  const RunDev* A;
  StepShared<TPB>* S;
  __device__ __forceinline__ void operator()(const Combined& x) const {
    if (threadIdx.x == ess_thread(TPB)) {
      S->ess = x.ess;
      S->resample = decide_resample(*A, x);
    }
    if (threadIdx.x == 0) {
      Q64 d, z0;
      long long tolZ;
      search_scalars(x, A->N, A->recip_n, S->uf, &d, &z0, &tolZ);
      S->scal[0] = d.hi;
      S->scal[1] = d.lo;
      S->scal[2] = z0.hi;
      S->scal[3] = z0.lo;
      S->scal[4] = (unsigned long long)tolZ;
    }
  }
};

// For a run combined in the last CTA of segment k: the decision and the closing
// (log Z, its records), and the next search's scalars, a thread each.
template <int TPB>
struct PublishRun {
  const RunDev* A;
  StepShared<TPB>* S;
  int k;
  __device__ __forceinline__ void operator()(const Combined& x) const {
    RunState* rs = A->rs;
    if (threadIdx.x == ess_thread(TPB)) {
      const bool resample = decide_resample(*A, x);
      rs->resample = resample ? 1 : 0;
      finish_segment(*A, k + 1, x, resample);
      rs->arrive = 0;
    }
    if (threadIdx.x == 0 && x.kmax != kDeadTile) {
      Q64 d, z0;
      long long tolZ;
      search_scalars(x, A->N, A->recip_n, S->uf, &d, &z0, &tolZ);
      rs->kmax = x.kmax;
      rs->G = x.G;
      rs->d_hi = d.hi;
      rs->d_lo = d.lo;
      rs->z0_hi = z0.hi;
      rs->z0_lo = z0.lo;
      rs->tolZ = tolZ;
    }
  }
};

// One tile of one run for segment k (the whole per-CTA body of a wave).
template <class M, int TPB>
__device__ __forceinline__ void step_tile(const RunDev& A, const int t, const int k,
                                          StepShared<TPB>& S, typename M::Lane& L, Stream& s,
                                          const bool early) {
  using R = typename M::R;
  RunState* rs = A.rs;
  const int N = A.N;
  const int i = t * A.tile + threadIdx.x;
  const bool valid = (int)threadIdx.x < A.tile && i < N;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int nb = k & 1, cb = nb ^ 1;
  const StateView Sc = A.state[cb];
  const StateView Sn = A.state[nb];
  const bool redundant = A.redundant != 0;
  // resuming a snapshot: segment resume_k - 1 loads the population instead of running it
  const bool load = A.resume_k > 0 && k == A.resume_k - 1;
  bool near = false;
  if (load) {
    if (valid) M::load(L, Sn, SnapView{A.snap_logw, A.snap_real, A.snap_int, A.snap_stack}, i, N, s);
  } else if (k > 0) {
    SearchCtx X;
    X.rec = A.rec[cb];
    bool resample;
    if (redundant) {
      // two threads form the decision and the search scalars, for all to read
      const Combined c = combine_offsets<TPB>(
          A.rec[cb], A.n_tiles, S.O, S.ks, S.red, A.ess ? A.tq[cb] : nullptr,
          PublishShared<TPB>{&A, &S});
      const bool go_on = c.kmax != kDeadTile && c.alive && k < A.max_segments;
      resample = S.resample != 0;
      // (closed by the tile's last thread: its warp is the one most often without particles)
      if (t == 0 && threadIdx.x == TPB - 1) {
        Combined x = c;
        x.ess = S.ess;
        finish_segment(A, k, x, resample);
      }
      if (!go_on) return;
      X.O = S.O;
      X.ks = S.ks;
      X.kmax = c.kmax;
      X.G = c.G;
      X.d = Q64{S.scal[0], S.scal[1]};
      X.z0 = Q64{S.scal[2], S.scal[3]};
      X.tolZ = (long long)S.scal[4];
    } else {
      resample = rs->resample != 0;
      X.O = A.tile_O;
      X.ks = nullptr;
      X.kmax = rs->kmax;
      X.G = rs->G;
      X.d = Q64{rs->d_hi, rs->d_lo};
      X.z0 = Q64{rs->z0_hi, rs->z0_lo};
      X.tolZ = rs->tolZ;
    }
    int a_s = i;
    if (resample && i - lane < N && (int)threadIdx.x - lane < A.tile) {  // (whole warps)
      const int i_last = min(N, (t + 1) * A.tile) - 1;
      a_s = systematic_search(min(i, i_last), t, A, X, A.E[cb], A.ends[cb], &near);
      near = near && valid;
    }
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
      if (bad) {  // the access is skipped: the particle is killed
        M::init(L);
        L.pc = PC_STOP;
        L.logw = neg_inf<R>();
      } else if (resample) {
        M::gather(L, Sc, Sn, a, i, N, A.md);
      } else {  // not resampled: the particle keeps its state and its accumulated weight
        M::gather(L, Sc, Sn, i, i, N, A.md);
        L.logw = (R)A.logw[i];
      }
    }
    warp_add_u64(&rs->n_near, near ? 1ull : 0ull);
  } else if (valid) {
    M::init(L);
  }
  if (SMC_DEBUG_CHECKS && valid && !(L.pc == PC_STOP || (L.pc >= 0 && L.pc < M::NB))) {
    debug_record(rs, 2, i);  // a block index outside the table: not dispatched
    L.pc = PC_STOP;
    L.logw = neg_inf<R>();
  }
  const bool active = valid && !load && L.pc != PC_STOP;
  const int n_exec = run_segment<M>(L, s, A.md, Sn, i, k, N, active);
  double lw = -INFINITY;
  int alive = 0;
  if (valid) {
    M::store(L, Sn, i, N);
    lw = widen(L.logw);
    A.logw[i] = lw;
    alive = L.pc != PC_STOP;
  }
  // Weights, first per warp as soon as the warp's particles reached the
  // checkpoint (overlapping the tile's slower warps): the warp's max M_w, its
  // power-of-two reference k_w = ceil(M_w / ln 2), and e_j = exp(logw_j - k_w
  // ln 2) 2^54 rounded to an integer on the integer pipes.  Then, after the tile barrier, the tile
  // reference k_t = max k_w, the exact shift of each weight to it, and the
  // tile's integer running sum E_j (the next segment's search keys).
  long long ef = 0;
  const double Mw = warp_max_key(lw);
  const int kw = is_neg_inf(Mw) ? kDeadTile : tile_exponent_fast(Mw);
  if (valid && kw != kDeadTile) {
    // (an FP32 log-weight is exact as a double, so both precisions share the
    // normaliser's integer-pipe exponential)
    if (kw > -2048 && kw < 2048) {
      ef = weight_fix54(lw, kw, ref_q58_lo(kw), A.md.tab);  // integer pipes only
    } else {
      const double kd = (double)kw;
      const double d = fma(-kd, kLn2Lo, fma(-kd, kLn2Hi, lw));  // lw - kw ln 2, two-part ln 2
      ef = exp_fix54(d, A.md.tab);
    }
  }
  // work counters: Philox blocks of the model's draw stream and blocks executed,
  // summed over the CTA: one atomic a CTA and counter.  (With one a warp, 65,536
  // of them fell on two words in a wave of 2^20 particles; that, a fence by every
  // thread and two more barriers took 20 of the rate-shift model's 178 us a wave.)
  // Kills are rare.
  // (a stopped particle's stream has moved only where a draw was taken ahead)
  const unsigned draws =
      __reduce_add_sync(0xffffffffu, (M::PREDRAW && early ? active : valid) ? s.d : 0u);
  const unsigned execs = __reduce_add_sync(0xffffffffu, (unsigned)n_exec);
  const unsigned kills = __reduce_add_sync(
      0xffffffffu, active ? (unsigned)L.overflow | ((unsigned)L.limited << 16) : 0u);
  if (lane == 0) {
    if (kills & 0xffffu) atomicAdd(&rs->n_overflow, (unsigned long long)(kills & 0xffffu));
    if (kills >> 16) atomicAdd(&rs->n_limit, (unsigned long long)(kills >> 16));
    S.kw[wid] = kw;
    S.draws[wid] = draws;
    S.execs[wid] = execs;
  }
  // The next wave's CTAs may start now (this one's particles are done): earlier
  // they would hold places on the SMs that other chains' CTAs can use, later their
  // start is not hidden.  At the CTA's start / here / at its end: batch of 512
  // 142.9 / 140.3 / 139.9 ms, CRBD 64k 24.2 / 24.0 / 24.5 us a wave, delayed
  // sampling 68.6 / 67.9 / 66.8, linear-Gaussian 23k 9.71 / 9.76 / 9.95.
  if (!early) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  alive = __syncthreads_or(alive);
  int kt = S.kw[0];
#pragma unroll
  for (int w = 1; w < TPB / 32; ++w) kt = max(kt, S.kw[w]);
  const int shift = kw == kDeadTile ? 64 : kt - kw;
  if (shift >= 63)
    ef = 0;
  else if (shift > 0)
    ef = (ef + (1ll << (shift - 1))) >> shift;
  const long long E = block_incl_scan_i64<32>(ef, nullptr);  // the warp's running sums
  if ((int)threadIdx.x < A.pad) A.E[nb][(size_t)t * A.pad + threadIdx.x] = E;
  if (A.ess) {  // the warp's sum of squared weights, units 2^-54 of 2^(2 k_t)
    const unsigned long long u = (unsigned long long)ef;
    unsigned long long sq = (__umul64hi(u, u) << 10) | ((u * u) >> 54);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
    if (lane == 0) S.sq[wid] = (long long)sq;
  }
  if (lane == 31) S.sum[wid] = E;
  __syncthreads();
  if (wid == TPB / 32 - 1) {  // the last warp closes the tile
    unsigned long long d = lane < TPB / 32 ? S.draws[lane] : 0u, x = lane < TPB / 32 ? S.execs[lane] : 0u;
    long long Q = A.ess && lane < TPB / 32 ? S.sq[lane] : 0;
#pragma unroll
    for (int o = TPB / 64; o > 0; o >>= 1) {
      d += __shfl_xor_sync(0xffffffffu, d, o);
      x += __shfl_xor_sync(0xffffffffu, x, o);
      Q += __shfl_xor_sync(0xffffffffu, Q, o);
    }
    // the warps' ends C_c (past the last warp: the tile's total) and the total
    long long C = lane < TPB / 32 ? S.sum[lane] : 0;
#pragma unroll
    for (int o = 1; o < TPB / 32; o <<= 1) {
      const long long y = __shfl_up_sync(0xffffffffu, C, o);
      if (lane >= o) C += y;
    }
    const long long total = __shfl_sync(0xffffffffu, C, TPB / 32 - 1);
    if (TPB > 32 && lane < 8) A.ends[nb][(size_t)t * 8 + lane] = lane < TPB / 32 ? C : total;
    if (lane == 0) {
      if (d) atomicAdd(&rs->n_draws, d);
      if (x) atomicAdd(&rs->n_blocks, x);
      if (A.ess) A.tq[nb][t] = Q;
    }
    __syncwarp();  // tq before the arrival
    if (lane == 31) {
      TileRec r;
      r.s = total;
      r.k = kt;
      r.alive = alive;
      A.rec[nb][t] = r;
      if (!redundant) {  // the run's last tile of the segment combines for the next wave
        __threadfence();
        const unsigned prev = atomicAdd(&rs->arrive, 1u);
        S.last = (prev == (unsigned)A.n_tiles - 1u);
      }
    }
  }
  if (redundant) return;  // the next wave combines
  __syncthreads();
  if (S.last) {  // the run's last tile of segment k: combine for the next wave
    __threadfence();
    const PublishRun<TPB> close{&A, &S, k};
    const Combined c = combine_offsets<TPB>(A.rec[nb], A.n_tiles, A.tile_O, nullptr, S.red,
                                            A.ess ? A.tq[nb] : nullptr, close);
    if (c.kmax == kDeadTile) close(c);
  }
}

constexpr unsigned kSms = 152;  // GB300's

// The block table of a model kind.
template <int KIND, typename R>
struct ModelOf;
template <typename R>
struct ModelOf<SMC_MODEL_LG, R> { using type = LgModel<R>; };
template <typename R>
struct ModelOf<SMC_MODEL_CRBD, R> { using type = TreeModel<R, false>; };
template <typename R>
struct ModelOf<SMC_MODEL_RATESHIFT, R> { using type = TreeModel<R, true>; };
template <typename R>
struct ModelOf<SMC_MODEL_GEOMETRIC, R> { using type = GeoModel<R>; };
template <typename R>
struct ModelOf<SMC_MODEL_SEIR, R> { using type = SeirModel<R>; };
template <typename R>
struct ModelOf<SMC_MODEL_CRBD_DS, R> { using type = TreeDsModel<R>; };

// Resident threads an SM that a wave kernel is bounded to.  A grid that fits at once
// with 768 (three CTAs of 256, 80 registers) is bound by each CTA's latency and wants
// the registers; a dense one by how many warps there are to switch between, and
// takes fewer.  us a wave, sparse / dense form: CRBD FP32 65,536 particles (456 CTAs)
// 16.4 / 19.8, 2^20 131.5 / 115.6, rate-shift FP32 2^20 145 / 126, CRBD FP64 65,536
// 20.5 / 23.1, 2^20 184 / 174, linear-Gaussian FP64 2^20 95 / 84, 23,171 7.23 / 7.43; a
// batch of 512 FP32 runs 152 / 128 ms with its CRBD runs in either form.  (FP32 waves
// of 2^20 linear-Gaussian particles stay at 1,024: 72 us, 75 with 1,280.)
template <typename R, int KIND>
__host__ __device__ constexpr int resident_threads(int tpb, bool dense) {
  if (!dense) return 768;
  if (sizeof(R) == 8 || (KIND == SMC_MODEL_LG && tpb == 256)) return 1024;
  return 1280;
}
__host__ __device__ constexpr int min_ctas(int threads, int tpb) {
  return threads / tpb < 32 ? threads / tpb : 32;
}

// One wave: CTA b runs tile cta_map[b].y of run cta_map[b].x, segment
// k = wave - start_wave of that run.
// KIND: the model (SMC_MODEL_*) that every run of the launch runs.
template <typename R, int TPB, int KIND, bool DENSE>
__global__ void __launch_bounds__(TPB, min_ctas(resident_threads<R, KIND>(TPB, DENSE), TPB))
    wave_kernel(const RunDev* __restrict__ runs, const int2* __restrict__ cta_map, unsigned wave,
                int alone) {
  __shared__ __align__(16) RunDev sr;
  __shared__ StepShared<TPB> S;
  const int2 rt = cta_map[blockIdx.x];
  {
    const int* src = reinterpret_cast<const int*>(runs + rt.x);
    int* dst = reinterpret_cast<int*>(&sr);
    for (int w = threadIdx.x; w < (int)(sizeof(RunDev) / 4); w += TPB) dst[w] = src[w];
  }
  __syncthreads();
  // Waves are launched with programmatic stream serialisation: a wave's CTAs may
  // start (and copy their run table, which no kernel writes) while the last CTAs
  // of the previous one still run; everything below reads what that wave wrote, so
  // it waits for its completion first.
  using M = typename ModelOf<KIND, R>::type;
  // (a lone chain's grid of at most one CTA an SM leaves room for the next wave's
  // CTAs beside its own: those then start at once, and what they do before the wait
  // is hidden.  Beside other chains they would take places from them)
  const bool early = alone && gridDim.x <= kSms;
  // (Triggered before the wait, several waves gather on the SMs, and the later ones take
  // the places that happen to come free, two CTAs of a wave on one SM beside idle ones:
  // SEIR FP32 with 122 CTAs of 128 195 us a day, after the wait 114; CRBD with delayed
  // sampling 30.7 / 24.3.  Only the models that draw ahead, whose blocks are short, are
  // faster so in CTAs of 256: nine sizes from 20,000 to 38,912 linear-Gaussian particles,
  // us a wave so / after the wait: FP64 all faster, 7.24 / 7.50 to 7.61 / 8.19; FP32 seven
  // faster, 6.80 / 6.86 to 7.01 / 7.17, two not (20,000 6.79 / 6.71, 31,000 6.75 / 6.66).)
  const bool ahead = early && M::PREDRAW && TPB == 256;
  if (ahead) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int k = (int)(wave - sr.start_wave);  // wraps correctly past 2^32 waves
  typename M::Lane L;
  Stream s{sr.k0, sr.k1, (uint32_t)(rt.y * sr.tile + threadIdx.x), (uint32_t)k, 0u, 0u, sr.md.tab};
  if constexpr (M::PREDRAW) {
    // (not for a segment that loads a snapshot, nor the one after it, which runs the
    // blocks that the snapshot names.  In larger grids most CTAs start
    // after the wave before them has ended: nothing to hide the draw behind, and
    // drawing there took a wave of 2^20 FP32 particles from 78 to 89 us)
    L.drawn = false;
    if (early && k > sr.resume_k && (int)threadIdx.x < sr.tile) M::predraw(L, s);
  }
  // the uniform of the search whose scalars this CTA may form, from the counter
  // alone: in the wait's shadow
  if (threadIdx.x == 0) S.uf = search_uniform(sr, sr.redundant ? k - 1 : k);
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (early && !ahead) asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  RunState* rs = sr.rs;
  if (*(volatile int32_t*)&rs->done || k < 0) return;
  step_tile<M, TPB>(sr, rt.y, k, S, L, s, early);
}

// One bucket of a wave, launched so that it may begin before the kernel ahead
// of it in the stream has finished (wave_kernel waits for it where it must).
template <typename R, int TPB, int KIND, bool DENSE>
cudaError_t launch_pdl(const RunDev* runs, const int2* map, int n, cudaStream_t st, unsigned wave,
                       bool alone) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)n);
  cfg.blockDim = dim3(TPB);
  cfg.dynamicSmemBytes = 0;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, wave_kernel<R, TPB, KIND, DENSE>, runs, map, wave, alone ? 1 : 0);
}

template <typename R, int KIND, bool DENSE>
cudaError_t launch_bucket(int b, const RunDev* runs, const int2* map, int n, cudaStream_t st,
                          unsigned wave, bool alone) {
  switch (b) {
    case 0: return launch_pdl<R, 32, KIND, DENSE>(runs, map, n, st, wave, alone);
    case 1: return launch_pdl<R, 64, KIND, DENSE>(runs, map, n, st, wave, alone);
    case 2: return launch_pdl<R, 128, KIND, DENSE>(runs, map, n, st, wave, alone);
    default: return launch_pdl<R, 256, KIND, DENSE>(runs, map, n, st, wave, alone);
  }
}

}  // namespace smc
