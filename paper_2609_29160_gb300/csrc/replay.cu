// Closed-loop replay (Sec. IV-B rescue and rebalance acting on live capacity,
// Sec. IV-C bounded transfer, Sec. VI-D actuation delays): the controller's
// moves change the servers that serve the requests, and the telemetry it
// scores comes from the requests as they are served.
//
// Readings (shared with the oracle's replay):
//  * each routable replica of a model is one server; a model's requests are
//    served in input order by whichever of its servers frees first; a request
//    needs d_first ms to its first token and d_total ms to its last once
//    started;
//  * window k is processed at T = (k+1)*win: every request that can start
//    before T starts first, then window k's telemetry (the window reduction's
//    token attribution and gauges) is scored with the smoothing carried over
//    windows, and on a control tick the controller acts on the replica counts
//    as they are;
//  * a transition commits at its tick; each donor replica it releases is the
//    donor's server that frees first: it takes no request from T on, finishes
//    the one it serves and returns its GPU sleep_ms after that; the receiver's
//    new server starts waking when its GPU is free (at T when the idle pool
//    paid, else when the transition's last released donor replica has
//    returned its GPU) and serves wake_ms later;
//  * a request not started by the end of the grid reports K*win for its
//    times; an invalid latent record reports -1 and is not served.
//
// GPU layout: one CTA per controller instance (a rescue threshold and a pacing
// cap). The servers only change on control ticks, so between two ticks the
// models are independent of each other: each warp takes a model's windows up to
// the next tick (at most 32 of them, one per lane) and
//   1. starts its requests in order. Only this is serial: a start takes the
//      server that frees first, a warp-wide minimum over free times held one
//      per lane (two or four for more servers);
//   2. attributes the started requests, one per lane, to the windows of a ring
//      in shared memory (windows beyond it in the workspace);
//   3. scores the windows, one per lane, with the smoothing chain passed from
//      lane to lane.
// On a tick one warp runs the controller with the models on its lanes. What
// bounds a replay is the start chain of its busiest model; up to 8 models a second
// warp takes the attribution off it. 160,000 requests of 8 models over 600 windows,
// 64 instances: 3.9 ms (4.9 with one warp a model, 7.7 when a start took two warp
// votes and a divergent write); a warp per
// instance with a lane per model (heaps of free times, attribution inside the
// start loop) took 78.3, 2,700 cycles a start.
#include <algorithm>

#include "common.cuh"
#include "internal.h"

namespace tre {
namespace {

constexpr unsigned kFull = 0xffffffffu;

// ---- latent records grouped by model, input order kept ----------------------
// One CTA per kGroupBlock records: valid model id per record (-1 when the record
// is not served), arrivals per (window, model), valid records per (block, model).
constexpr int kGroupBlock = 1024;
__global__ void __launch_bounds__(kGroupBlock)
k_rp_valid(ReplayLatent lat, int M, FastDiv fwin, int64_t span, int8_t* __restrict__ vm,
           int32_t* __restrict__ arr_cnt, int32_t* __restrict__ blk_cnt) {
  __shared__ int32_t cnt[64];
  if (threadIdx.x < M) cnt[threadIdx.x] = 0;
  __syncthreads();
  const int64_t i = (int64_t)blockIdx.x * kGroupBlock + threadIdx.x;
  if (i < lat.n) {
    const int m = lat.model[i];
    const int ta = lat.t_arr[i], df = lat.d_first[i];
    const bool ok = m >= 0 && m < M && ta >= 0 && ta < span && df >= 0 && lat.d_total[i] >= df &&
                    lat.L_in[i] >= 0 && lat.L_out[i] >= 1;
    vm[i] = ok ? (int8_t)m : (int8_t)-1;
    if (ok) {
      atomicAdd(&arr_cnt[(size_t)fwin.div((uint32_t)ta) * M + m], 1);
      atomicAdd(&cnt[m], 1);
    }
  }
  __syncthreads();
  if (threadIdx.x < M) blk_cnt[(size_t)blockIdx.x * M + threadIdx.x] = cnt[threadIdx.x];
}

// one warp per model (warp w takes models w, w + 32, ...): exclusive prefix of
// its block counts, then the models' offsets in the grouped order
__global__ void __launch_bounds__(1024)
k_rp_offsets(int M, int n_blk, int32_t* __restrict__ blk_cnt, int32_t* __restrict__ base) {
  __shared__ int32_t total[64];
  const int lane = threadIdx.x & 31;
  for (int m = threadIdx.x >> 5; m < M; m += 32) {
    int32_t run = 0;
    for (int b0 = 0; b0 < n_blk; b0 += 32) {
      const int b = b0 + lane;
      const int32_t v = b < n_blk ? blk_cnt[(size_t)b * M + m] : 0;
      int32_t inc = v;
      for (int o = 1; o < 32; o <<= 1) {
        const int32_t x = __shfl_up_sync(kFull, inc, o);
        if (lane >= o) inc += x;
      }
      if (b < n_blk) blk_cnt[(size_t)b * M + m] = run + inc - v;
      run += __shfl_sync(kFull, inc, 31);
    }
    if (lane == 0) total[m] = run;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    int32_t b = 0;
    for (int m = 0; m < M; ++m) {
      base[m] = b;
      b += total[m];
    }
    base[M] = b;
  }
}

// the model-grouped columns a lane walks: arrival, time to first and last
// token, index; prompt and output lengths. A record's place among its model's
// records of the block is counted within the warp and over the warps before it.
__global__ void __launch_bounds__(kGroupBlock)
k_rp_group(ReplayLatent lat, int M, const int8_t* __restrict__ vm,
           const int32_t* __restrict__ blk_off, const int32_t* __restrict__ base,
           int4* __restrict__ g) {
  __shared__ int32_t wcnt[kGroupBlock / 32][64];
  const int64_t i = (int64_t)blockIdx.x * kGroupBlock + threadIdx.x;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  for (int c = threadIdx.x; c < (kGroupBlock / 32) * 64; c += kGroupBlock) wcnt[c >> 6][c & 63] = 0;
  __syncthreads();
  const int m = i < lat.n ? vm[i] : -1;
  const unsigned same = __match_any_sync(kFull, m);
  const int before = __popc(same & ((1u << lane) - 1u));
  if (m >= 0 && before == 0) wcnt[wid][m] = __popc(same);
  __syncthreads();
  if (m < 0) return;
  int32_t p = base[m] + blk_off[(size_t)blockIdx.x * M + m] + before;
  for (int w = 0; w < wid; ++w) p += wcnt[w][m];
  g[2 * (size_t)p] = make_int4(lat.t_arr[i], lat.d_first[i], lat.d_total[i], (int32_t)i);
  g[2 * (size_t)p + 1] = make_int4(lat.L_in[i], lat.L_out[i], 0, 0);
}

// served records start as "not started" (K*win) or "not served" (-1)
__global__ void k_rp_init_records(int64_t n, int n_inst, int32_t span, const int8_t* __restrict__ vm,
                                  int32_t* ts, int32_t* tf, int32_t* te) {
  const int64_t total = n * n_inst;
  for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < total;
       x += (int64_t)gridDim.x * blockDim.x) {
    const int32_t v = vm[x % n] >= 0 ? span : -1;
    ts[x] = v;
    tf[x] = v;
    te[x] = v;
  }
}

// ---- the replay ------------------------------------------------------------
// Per-model window ring (power of two) and the counts a window collects. A
// segment is at most 32 windows, so a ring of 64 holds every window a request
// started in the segment can reach within 32 windows of its end.
constexpr int kRing = 64;
enum { kP = 0, kD = 1, kEnd = 2, kLate = 3, kStart = 4, kCounts = 5 };
constexpr int kFarCounts = 4;        // a start is never beyond its own segment
constexpr int kMaxWarps = 16;        // models of an instance take turns beyond this
constexpr int kMaxPairs = 8;         // models with two warps each
// a server's free time as an unsigned 32-bit millisecond; later ones (wake and
// sleep delays near 2^31) are kept at kNever, past the end of every grid
constexpr uint32_t kNever = 0xfffffffeu, kNoServer = 0xffffffffu;

__device__ __forceinline__ uint32_t free_at(long long t) {
  return t < (long long)kNever ? (uint32_t)t : kNever;
}

// first window at or after k that ends a tick of cadence c (a multiple of c
// falls in (k*win, (k+1)*win]): the window of the next multiple above k*win
__device__ __forceinline__ int next_tick(int k, uint32_t win, uint32_t c) {
  const unsigned long long t = ((unsigned long long)k * win / c + 1) * c;
  const unsigned long long w = (t + win - 1) / win - 1;
  return w < 0x7fffffffull ? (int)w : 0x7fffffff;
}

__device__ __forceinline__ uint32_t key_order(float z) {
  const uint32_t u = __float_as_uint(z);
  return u == 0x80000000u ? 0x80000000u : u ^ ((u >> 31) ? 0xffffffffu : 0x80000000u);
}
__device__ __forceinline__ unsigned long long key_order(double z) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(z);
  return u == 0x8000000000000000ull ? u : u ^ ((u >> 63) ? ~0ull : 0x8000000000000000ull);
}

// Lowest (MAX: highest) value among the lanes of `elig`, -1 when there is none,
// as an ascending scan finds it: the first lane of equal ones; a NaN only when
// it is the first eligible one.
template <bool MAX, class T>
__device__ __forceinline__ int best_lane(unsigned elig, T z) {
  if (!elig) return -1;
  const unsigned num = elig & ~__ballot_sync(kFull, z != z);
  const int first = __ffs(elig) - 1;
  if (!(num >> first & 1u)) return first;
  const int lane = threadIdx.x & 31;
  const auto key = MAX ? ~key_order(z) : key_order(z);
  bool in = num >> lane & 1u;
  if (sizeof(T) == 8) {
    const uint32_t hi = (uint32_t)((unsigned long long)key >> 32);
    const uint32_t mh = __reduce_min_sync(kFull, in ? hi : 0xffffffffu);
    in = in && hi == mh;
  }
  const uint32_t lo = (uint32_t)key;
  const uint32_t ml = __reduce_min_sync(kFull, in ? lo : 0xffffffffu);
  return __ffs(__ballot_sync(kFull, in && lo == ml)) - 1;
}

// The same over up to 64 models, two per lane (z[0] models 0-31, z[1] 32-63)
template <bool MAX, class T>
__device__ __forceinline__ int best_model(const unsigned (&elig)[2], const T (&z)[2]) {
  const int a = best_lane<MAX>(elig[0], z[0]);
  const int c = best_lane<MAX>(elig[1], z[1]);
  if (a < 0) return c < 0 ? -1 : 32 + c;
  if (c < 0) return a;
  const T za = __shfl_sync(kFull, z[0], a), zc = __shfl_sync(kFull, z[1], c);
  // a NaN first in the upper half stays out when the lower half has a model
  if (zc == zc) return (MAX ? zc > za : zc < za) ? 32 + c : a;
  const unsigned num = elig[1] & ~__ballot_sync(kFull, z[1] != z[1]);
  const int c2 = best_lane<MAX>(num, z[1]);
  if (c2 < 0) return a;
  const T z2 = __shfl_sync(kFull, z[1], c2);
  return (MAX ? z2 > za : z2 < za) ? 32 + c2 : a;
}

// A model's servers in shared memory (or the workspace), unordered; the warp
// finds the one that frees first.
struct Servers {
  uint32_t* v;
  int n;
  __device__ __forceinline__ uint32_t first(int& at) const {
    const int lane = threadIdx.x & 31;
    uint32_t best = kNoServer;
    int i = -1;
    for (int q = lane; q < n; q += 32)
      if (v[q] < best) {
        best = v[q];
        i = q;
      }
    const uint32_t f = __reduce_min_sync(kFull, best);
    const int src = __ffs(__ballot_sync(kFull, best == f)) - 1;
    at = __shfl_sync(kFull, i, src);
    return f;
  }
};

// what a model carries from segment to segment
template <class T> struct ModelState {
  int32_t head, end;
  uint32_t arrived, started, ended;   // running totals (differences are exact modulo 2^32)
  int32_t far_hi;                     // last window with counts in the workspace
  int32_t init;
  unsigned long long met;
  T S;
};

// Starts a model's requests in order until one cannot start before t_end, its
// servers' free times in registers, R per lane. Calls `done(st, c0, c1)` with the
// lanes' started requests, up to 32 at a time (st = kNoServer: none). A server is
// a key: its free time since the earliest one, with its number in the low bits, so
// that one warp minimum finds both the time and the server, and a start is a chain
// of a minimum, a maximum, a sum and a select without a branch (two warp votes and
// a divergent write of the server took 250 cycles a start). Times kLate and more
// past the earliest one are all "late"; returns false, with nothing done, when
// t_end itself lies past that (37 hours up to 32 servers, nine above 64).
template <int R, class F>
__device__ __forceinline__ bool start_requests(uint32_t* sv, int n, const int4* __restrict__ grp,
                                               int& head, int end, uint32_t t_end, F&& done) {
  constexpr int kBits = R == 1 ? 5 : R == 2 ? 6 : 7;
  constexpr uint32_t kLate = (1u << (32 - kBits)) - 2;
  static_assert(R <= 4, "a server's number has seven bits");
  const int lane = threadIdx.x & 31;
  uint32_t s[R], key[R], low = kNoServer;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    s[r] = lane + 32 * r < n ? sv[lane + 32 * r] : kNoServer;
    low = min(low, s[r]);
  }
  const uint32_t t0 = __reduce_min_sync(kFull, low);
  if (t0 >= t_end) return true;
  const uint32_t stop = t_end - t0;
  if (stop > kLate) return false;
#pragma unroll
  for (int r = 0; r < R; ++r)
    key[r] = lane + 32 * r < n ? (min(s[r] - t0, kLate) << kBits) + (uint32_t)(lane + 32 * r)
                               : kNoServer;
  auto fetch = [&](int p, int4& a, int4& c) {
    if (p < end) {
      a = __ldg(&grp[2 * (size_t)p]);
      c = __ldg(&grp[2 * (size_t)p + 1]);
    }
  };
  int4 c0 = make_int4(0, 0, 0, 0), c1 = c0, n0 = c0, n1 = c0;
  fetch(head + lane, c0, c1);
  bool go = head < end;
  while (go) {
    fetch(head + 32 + lane, n0, n1);               // the next 32, behind this batch's chain
    // past the last request: one that arrives too late
    const uint32_t arr = head + lane < end
                             ? min((uint32_t)c0.x > t0 ? (uint32_t)c0.x - t0 : 0u, kLate) : kLate;
    uint32_t mine = kNoServer;
    for (int j8 = 0; j8 < 32 && go; j8 += 8) {
#pragma unroll
      for (int j = j8; j < j8 + 8; ++j) {
        const uint32_t ta = __shfl_sync(kFull, arr, j);
        const uint32_t dt = (uint32_t)__shfl_sync(kFull, c0.z, j);
        uint32_t first = key[0];
#pragma unroll
        for (int r = 1; r < R; ++r) first = min(first, key[r]);
        first = __reduce_min_sync(kFull, first);
        const uint32_t st = max(first >> kBits, ta);
        go = go && st < stop;
        const uint32_t te = min(st + dt, kLate);
#pragma unroll
        for (int r = 0; r < R; ++r)
          if (go && key[r] == first) {
            key[r] = (te << kBits) + (uint32_t)(lane + 32 * r);
            s[r] = min(t0 + st + dt, kNever);
          }
        if (go && lane == j) mine = t0 + st;
      }
    }
    head += __popc(__ballot_sync(kFull, mine != kNoServer));
    if (__any_sync(kFull, mine != kNoServer)) done(mine, c0, c1);
    go = go && head < end;
    c0 = n0;
    c1 = n1;
  }
#pragma unroll
  for (int r = 0; r < R; ++r)
    if (lane + 32 * r < n) sv[lane + 32 * r] = s[r];
  return true;
}

// the same with the free times left in memory, for more servers than four per
// lane and for longer stretches of time. A start reads all free times up to
// kScanServers; above (BLOCKS) the earliest one of each of up to 256 blocks of
// servers is kept eight per lane, and a start reads one block. 20,000 requests of 2
// models in 60 windows: 200 servers a model 2.62 ms by reading all, 3.23 by blocks;
// 600 servers 3.21 and 3.21; 1,000 servers 5.13 and 3.22; 32,768 servers 112 and 4.0.
constexpr int kScanServers = 600;
template <bool BLOCKS, class F>
__device__ __forceinline__ void start_requests_mem(uint32_t* sv, int n,
                                                   const int4* __restrict__ grp, int& head,
                                                   int end, uint32_t t_end, F&& done) {
  constexpr int R = BLOCKS ? 8 : 1;
  const int lane = threadIdx.x & 31;
  bool more = head < end;
  if (!more || (uint32_t)__ldg(&grp[2 * (size_t)head]).x >= t_end) return;
  const int len = ((n + 32 * R - 1) / (32 * R) + 31) / 32 * 32;   // of a block
  uint32_t low[R];                       // of block r * 32 + lane
  if constexpr (BLOCKS) {
#pragma unroll
    for (int r = 0; r < R; ++r) {
      low[r] = kNoServer;
#pragma unroll 4
      for (int i = 0; i < 32; ++i) {
        const int q0 = (r * 32 + i) * len, q1 = min(q0 + len, n);
        uint32_t v = kNoServer;
        for (int q = q0 + lane; q < q1; q += 32) v = min(v, sv[q]);
        v = __reduce_min_sync(kFull, v);
        if (i == lane) low[r] = v;
      }
    }
  }
  while (more) {
    int4 c0 = make_int4(0, 0, 0, 0), c1 = c0;
    if (head + lane < end) {
      c0 = __ldg(&grp[2 * (size_t)(head + lane)]);
      c1 = __ldg(&grp[2 * (size_t)(head + lane) + 1]);
    }
    const int cnt = min(32, end - head);
    uint32_t mine = kNoServer;
    int j = 0;
    for (; j < cnt; ++j) {
      const uint32_t ta = (uint32_t)__shfl_sync(kFull, c0.x, j);
      const uint32_t dt = (uint32_t)__shfl_sync(kFull, c0.z, j);
      uint32_t st;
      if constexpr (BLOCKS) {
        uint32_t l = low[0];
        int lr = 0;
#pragma unroll
        for (int r = 1; r < R; ++r)
          if (low[r] < l) {
            l = low[r];
            lr = r;
          }
        const uint32_t first = __reduce_min_sync(kFull, l);
        st = max(ta, first);
        if (st >= t_end) break;
        const int owner = __ffs(__ballot_sync(kFull, l == first)) - 1;
        const int blk = __shfl_sync(kFull, lr, owner) * 32 + owner;
        // the block's first server, and the block's minimum with its new free time
        uint32_t best = kNoServer, next = kNoServer;
        int at = -1;
        for (int q = blk * len + lane; q < min((blk + 1) * len, n); q += 32) {
          const uint32_t v = sv[q];
          next = min(next, max(v, best));
          if (v < best) {
            best = v;
            at = q;
          }
        }
        const uint32_t te = min(st + dt, kNever);
        if (lane == __ffs(__ballot_sync(kFull, best == first)) - 1) {
          sv[at] = te;
          best = min(next, te);
        }
        __syncwarp();
        const uint32_t left = __reduce_min_sync(kFull, best);
#pragma unroll
        for (int r = 0; r < R; ++r)
          if (blk == r * 32 + lane) low[r] = left;
      } else {
        int at;
        st = max(ta, Servers{sv, n}.first(at));
        if (st >= t_end) break;
        __syncwarp();
        if (lane == 0) sv[at] = min(st + dt, kNever);
        __syncwarp();
      }
      if (lane == j) mine = st;
    }
    head += j;
    if (j > 0) done(mine, c0, c1);
    more = j == 32 && head < end;
  }
}

__device__ __forceinline__ uint32_t warp_scan(uint32_t v) {
  const int lane = threadIdx.x & 31;
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t x = __shfl_up_sync(kFull, v, o);
    if (lane >= o) v += x;
  }
  return v;
}

// both warps of a pair (barrier 0 is the block's)
__device__ __forceinline__ void pair_sync(int pair) {
  asm volatile("bar.sync %0, 64;" :: "r"(pair + 1) : "memory");
}

// PAIR: two warps per model, one that runs the start chain and one that attributes
// the batch before and scores. They swap batches of 32 starts through two buffers
// and meet once a batch, so a batch costs the longer of the two.
template <class T, bool PAIR>
__global__ void __launch_bounds__(32 * kMaxWarps)
k_replay(const __grid_constant__ ReplayBatch<T> b) {
  extern __shared__ __align__(16) unsigned char rsm[];
  __shared__ uint32_t s_batch[PAIR ? kMaxPairs : 1][2][32];   // start times
  __shared__ int32_t s_more[PAIR ? kMaxPairs : 1][2];         // a batch follows
  __shared__ int32_t s_head[PAIR ? kMaxPairs : 1];            // next request to start
  const int lane = threadIdx.x & 31;
  const int n_warps = (blockDim.x >> 5) / (PAIR ? 2 : 1);
  const bool starts = PAIR && (int)(threadIdx.x >> 5) >= n_warps;
  const int wid = (int)(threadIdx.x >> 5) - (starts ? n_warps : 0);
  int buf = 0;
  const int inst = blockIdx.x;
  const int M = b.M, K = b.K;
  const uint32_t win = (uint32_t)b.win;
  const FastDiv fwin(win);
  const uint32_t span = (uint32_t)K * win;
  // shared memory: model states, Z row, replicas, server counts, class and flag
  // rows, rings, free times (when they fit)
  ModelState<T>* st_m = reinterpret_cast<ModelState<T>*>(rsm);
  T* zrow = reinterpret_cast<T*>(st_m + M);
  int32_t* rep = reinterpret_cast<int32_t*>(zrow + M);
  int32_t* n_srv = rep + M;
  uint8_t* crow = reinterpret_cast<uint8_t*>(n_srv + M);
  uint8_t* frow = crow + M;                     // bit 0: guard breached; bit 1: lost capacity
  uint32_t* ring = reinterpret_cast<uint32_t*>(rsm + b.ring_off);    // [kCounts][M][kRing]
  uint32_t* srv = b.gsrv ? b.gsrv + (size_t)inst * M * b.hcap
                         : reinterpret_cast<uint32_t*>(rsm + b.srv_off);   // [M][hcap]
  const int ti = inst / b.n_cap, ci = inst % b.n_cap;
  const int pacing = b.cap_list[ci];
  // later windows' prompt tokens, decode tokens, running-span ends and late
  // first tokens, [4][K + 1][M]
  uint32_t* far = b.acc + (size_t)inst * kFarCounts * (K + 1) * M;
  const size_t far_arr = (size_t)(K + 1) * M;
  for (int c = threadIdx.x; c < kCounts * M * kRing; c += blockDim.x) ring[c] = 0;
  for (int m = threadIdx.x; m < M; m += blockDim.x) {
    ModelState<T>& s = st_m[m];
    s.head = b.base[m];
    s.end = b.base[m + 1];
    s.arrived = s.started = s.ended = 0;
    s.far_hi = -1;
    s.init = 0;
    s.met = 0;
    s.S = (T)0;
    if (PAIR) s_head[m] = b.base[m];
    rep[m] = b.r0[m];
    n_srv[m] = max(b.r0[m], 0);
  }
  // initial replicas; every warp forms the sum itself
  long long used = 0;
  bool bad = false;
  for (int m = lane; m < M; m += 32) {
    const int32_t r0 = b.r0[m], g = b.footprint[m];
    bad |= r0 < 0 || g < 1 || b.r_min[m] < 0;
    used += (long long)g * r0;
  }
  for (int o = 16; o > 0; o >>= 1) used += __shfl_xor_sync(kFull, used, o);
  if (__any_sync(kFull, bad) || used > b.budget) {
    if (threadIdx.x == 0) {
      b.diag->err = TRE_EINVAL;
      b.n_moves[inst] = 0;
    }
    return;
  }
  __syncthreads();
  // one server free at t = 0 per replica
  for (int m = wid; m < M; m += n_warps)
    for (int q = lane; q < n_srv[m]; q += 32) srv[(size_t)m * b.hcap + q] = 0;
  // the controller's state (the first warp's copy is the live one)
  long long pool = b.budget - used, reb_until = 0;
  int64_t nm = 0;
  const T dt = div_rn(from_i32<T>(b.win), (T)1000);
  __syncthreads();

  for (int k0 = 0; k0 < K;) {
    // the segment: windows k0 .. k1, up to the next tick, at most 32
    const int tick = min(next_tick(k0, win, (uint32_t)b.fast_ms),
                         next_tick(k0, win, (uint32_t)b.slow_ms));
    const int k1 = min(min(tick, k0 + 31), K - 1);
    const int n_win = k1 - k0 + 1;
    const uint32_t t_end = (uint32_t)(k1 + 1) * win;
    auto start = [&](int m, int& head, int end, auto&& done) {
      const int n = n_srv[m];
      uint32_t* sv = srv + (size_t)m * b.hcap;
      if (n <= 0 || head >= end) return;
      const bool held =
          n <= 32    ? start_requests<1>(sv, n, b.grp, head, end, t_end, done)
          : n <= 64  ? start_requests<2>(sv, n, b.grp, head, end, t_end, done)
          : n <= 128 ? start_requests<4>(sv, n, b.grp, head, end, t_end, done)
                     : false;
      if (!held) {
        if (n <= kScanServers) start_requests_mem<false>(sv, n, b.grp, head, end, t_end, done);
        else start_requests_mem<true>(sv, n, b.grp, head, end, t_end, done);
      }
    };
    if (starts) {
      auto pass = [&](uint32_t st, bool more) {
        if (more) s_batch[wid][buf][lane] = st;
        if (lane == 0) s_more[wid][buf] = more;
        pair_sync(wid);
        buf ^= 1;
      };
      for (int m = wid; m < M; m += n_warps) {
        int head = s_head[m];
        start(m, head, b.base[m + 1],
              [&](uint32_t st, const int4&, const int4&) { pass(st, true); });
        pass(kNoServer, false);
        if (lane == 0) s_head[m] = head;
        __syncwarp();
      }
    } else for (int m = wid; m < M; m += n_warps) {
      ModelState<T>& s = st_m[m];
      uint32_t* my_ring = ring + (size_t)m * kRing;
      int head = s.head;
      const int end = s.end, head0 = head;
      int far_hi = -1;
      unsigned met = 0;
      int k_now = k0;                           // the window the last start was processed in
      const long long slo = b.slo_ms ? (long long)b.slo_ms[m] : -1;
      const long long guard = b.guard_ms ? (long long)b.guard_ms[m] : 0;
      auto add = [&](int arr, int kt, uint32_t v) {
        if (kt - k0 < kRing) {
          atomicAdd(&my_ring[(size_t)arr * M * kRing + (kt & (kRing - 1))], v);
        } else {
          atomicAdd(&far[arr * far_arr + (size_t)kt * M + m], v);
          far_hi = max(far_hi, kt);
        }
      };
      auto done = [&](uint32_t st, const int4& c0, const int4& c1) {
        // a request is processed in the window of its start, or in that of the
        // one before it where arrivals are out of order; what it would add to
        // windows already scored is not seen
        const bool on = st != kNoServer;
        int kp = on ? (int)fwin.div(st) : 0;
        for (int o = 1; o < 32; o <<= 1) {
          const int x = __shfl_up_sync(kFull, kp, o);
          if (lane >= o) kp = max(kp, x);
        }
        kp = max(kp, k_now);
        k_now = __shfl_sync(kFull, kp, 31);
        if (!on) return;
        const uint32_t ta = (uint32_t)c0.x;
        const uint32_t tf = min(st + (uint32_t)c0.y, 2147483647u);
        const uint32_t te = min(st + (uint32_t)c0.z, 2147483647u);
        const uint32_t L = (uint32_t)c1.y;
        if (b.o_ts) {
          const size_t x = (size_t)inst * b.lat.n + c0.w;
          b.o_ts[x] = (int32_t)st;
          b.o_tf[x] = (int32_t)tf;
          b.o_te[x] = (int32_t)te;
        }
        const long long ttft = (long long)tf - (long long)ta;
        met += b.slo_ms && ttft <= slo;
        add(kStart, kp, 1u);
        const int ke = (int)fwin.div(te);
        if (tf < span) {
          const int kf = (int)fwin.div(tf);
          // tokens of the first-token window, then a window at a time without
          // dividing: one window on adds win * (L - 1) = Q * dur + R
          uint32_t tok = L, rem = 0, Q = 0, R = 0;
          const uint32_t dur = te - tf;
          const bool later = L > 1 && ke > kf;
          if (later) {
            unsigned long long q, r;
            divmod((unsigned long long)((uint32_t)(kf + 1) * win - tf) * (L - 1), dur, q, r);
            tok = (uint32_t)q + (r != 0);
            rem = r ? (uint32_t)r - 1 : dur - 1;
            if (ke > kf + 1) {                  // dur > win here
              divmod((unsigned long long)win * (L - 1), dur, q, r);
              Q = (uint32_t)q;
              R = (uint32_t)r;
            }
          }
          if (kf >= kp) {
            if (b.guard_ms && ttft > guard) add(kLate, kf, 1u);
            if (c1.x) add(kP, kf, (uint32_t)c1.x);
            if (tok) add(kD, kf, tok);
          }
          if (later) {
            const int k_full = min(ke - 1, K - 1);
            for (int k = kf + 1; k <= k_full; ++k) {
              const uint32_t t = rem + R, c = t >= dur ? 1u : 0u;
              rem = t - (c ? dur : 0u);
              const uint32_t d = Q + c;
              tok += d;
              if (d && k >= kp) add(kD, k, d);
            }
            if (ke < K && L != tok && ke >= kp) add(kD, ke, L - tok);
          }
        }
        // the running span ends in window te / win (never read past the grid)
        if (te < span && ke >= kp) add(kEnd, ke, 1u);
      };
      if (PAIR) {
        auto fetch = [&](int q, int4& x, int4& y) {
          if (q < end) {
            x = __ldg(&b.grp[2 * (size_t)q]);
            y = __ldg(&b.grp[2 * (size_t)q + 1]);
          }
        };
        int4 c0 = make_int4(0, 0, 0, 0), c1 = c0, x0 = c0, x1 = c0;
        fetch(head + lane, c0, c1);
        while (true) {
          fetch(head + 32 + lane, x0, x1);
          pair_sync(wid);
          const bool more = s_more[wid][buf] != 0;
          const uint32_t st = s_batch[wid][buf][lane];
          buf ^= 1;
          if (!more) break;
          head += __popc(__ballot_sync(kFull, st != kNoServer));
          done(st, c0, c1);
          c0 = x0;
          c1 = x1;
        }
      } else {
        start(m, head, end, done);
      }
      __syncwarp();
      // the segment's windows, one per lane
      const int k = k0 + lane;
      const bool in = lane < n_win;
      uint32_t v[kCounts] = {0, 0, 0, 0, 0};
      const int fh = max(s.far_hi, (int)__reduce_max_sync(kFull, far_hi));
      if (fh > s.far_hi) __threadfence();       // far counts are read segments later
      if (in) {
#pragma unroll
        for (int a = 0; a < kCounts; ++a) {
          uint32_t* slot = &my_ring[(size_t)a * M * kRing + (k & (kRing - 1))];
          v[a] = *slot;
          *slot = 0;
        }
        if (k <= s.far_hi) {
#pragma unroll
          for (int a = 0; a < kFarCounts; ++a) v[a] += __ldcg(&far[a * far_arr + (size_t)k * M + m]);
        }
      }
      const uint32_t arr = warp_scan(in ? (uint32_t)b.arr_cnt[(size_t)k * M + m] : 0u) + s.arrived;
      const uint32_t started = warp_scan(v[kStart]) + s.started;
      const uint32_t ended = warp_scan(v[kEnd]) + s.ended;
      const int32_t P = (int32_t)v[kP], D = (int32_t)v[kD];
      const int32_t A = (int32_t)(started - ended), W = (int32_t)(arr - started);
      const bool idle = !in || (P == 0 && D == 0 && A == 0 && W == 0);
      T raw = (T)0;
      if (!idle) {
        const T num = add_rn(mul_rn(b.w_p[m], div_rn(from_i32<T>(P), dt)),
                             div_rn(from_i32<T>(D), dt));
        T den = add_rn(from_i32<T>(A), mul_rn(b.w_q[m], from_i32<T>(W)));
        if (den < (T)1) den = (T)1;
        raw = div_rn(num, den);
      }
      const unsigned live = __ballot_sync(kFull, !idle);
      const T al = b.alpha[m], be = (T)1 - al;
      const T ar = mul_rn(al, raw);
      T S = s.S, mine = (T)0;
      int init = s.init;
      for (int w = 0; w < n_win; ++w) {
        const T x1 = __shfl_sync(kFull, ar, w), r1 = __shfl_sync(kFull, raw, w);
        if (live >> w & 1u) {
          S = init ? add_rn(x1, mul_rn(be, S)) : r1;
          init = 1;
        }
        if (lane == w) mine = S;
      }
      const T Z = div_rn(mine, b.theta[m]);
      uint8_t cl;
      if (idle) cl = kIdle;
      else if (Z < (b.n_tau > 0 ? b.tau_list[ti] : b.tau_crit[m])) cl = kCrit;
      else if (Z > b.tau_surp[m]) cl = kSurp;
      else cl = kNom;
      if (in && b.Z) {
        const size_t y = ((size_t)inst * K + k) * M + m;
        b.Z[y] = Z;
        b.cls[y] = cl;
      }
      if (lane == n_win - 1) {
        zrow[m] = Z;
        crow[m] = cl;
        // latency guard breached in the window; requests waiting with no
        // routable replica (lost capacity)
        frow[m] = (uint8_t)((b.guard_ms && v[kLate] ? 1 : 0) | (rep[m] == 0 && W > 0 ? 2 : 0));
      }
      const uint32_t a1 = __shfl_sync(kFull, arr, n_win - 1);
      const uint32_t s1 = __shfl_sync(kFull, started, n_win - 1);
      const uint32_t e1 = __shfl_sync(kFull, ended, n_win - 1);
      const unsigned mt = b.slo_ms && head > head0 ? __reduce_add_sync(kFull, met) : 0u;
      if (lane == 0) {
        s.head = head;
        s.arrived = a1;
        s.started = s1;
        s.ended = e1;
        s.far_hi = fh;
        s.met += mt;
        s.S = S;
        s.init = init;
      }
      __syncwarp();
    }
    const int k = k1;
    k0 = k1 + 1;
    if (k != tick) continue;                    // no tick in the segment's last window
    __syncthreads();
    if (wid == 0 && !starts) {
      const long long Tk = (long long)t_end;
      const bool fast = next_tick(k, win, (uint32_t)b.fast_ms) == k;
      const bool slow = next_tick(k, win, (uint32_t)b.slow_ms) == k;
      // models on lanes, two per lane
      T z[2];
      uint8_t rg[2];
      bool held[2];
      int32_t r[2], rmin[2], fp[2];
      unsigned idle_m[2], surp_m[2], nom_m[2], crit_m[2], breach[2], lost[2];
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const int m = lane + 32 * j;
        const bool has = m < M;
        z[j] = has ? zrow[m] : (T)0;
        const uint8_t c = has ? crow[m] : kIdle, f = has ? frow[m] : (uint8_t)0;
        held[j] = f & 1;
        r[j] = has ? rep[m] : 0;
        rmin[j] = has ? b.r_min[m] : 0;
        fp[j] = has ? b.footprint[m] : 0;
        rg[j] = !has ? (uint8_t)0xff
                : c == kIdle ? kIdle
                : z[j] < (b.n_tau > 0 ? b.tau_list[ti] : b.tau_crit[m]) ? kCrit
                : z[j] > b.tau_surp[m] ? kSurp : kNom;
        idle_m[j] = __ballot_sync(kFull, rg[j] == kIdle);
        surp_m[j] = __ballot_sync(kFull, rg[j] == kSurp);
        nom_m[j] = __ballot_sync(kFull, rg[j] == kNom);
        crit_m[j] = __ballot_sync(kFull, rg[j] == kCrit);
        breach[j] = __ballot_sync(kFull, f & 1);
        lost[j] = __ballot_sync(kFull, (f & 2) != 0);
      }
      auto value = [&](const T (&a)[2], int m) -> T {
        return __shfl_sync(kFull, m < 32 ? a[0] : a[1], m & 31);
      };
      auto count = [&](const int32_t (&a)[2], int m) -> int32_t {
        return __shfl_sync(kFull, m < 32 ? a[0] : a[1], m & 31);
      };
      int recv = -1, kind = 0;
      bool nom_above = false, deferred = false;
      if (fast) {
        // rescue: a latency-guard breach pre-empts every other event (lowest
        // Z among the breaching models); otherwise the lowest Z among critical
        // models and models that lost their routable capacity. A rebalance
        // transfer in progress defers a rescue without a breach; the pending
        // rescue keeps the slow loop out of the tick.
        const bool hard = (breach[0] | breach[1]) != 0;
        const unsigned want[2] = {hard ? breach[0] : crit_m[0] | lost[0],
                                  hard ? breach[1] : crit_m[1] | lost[1]};
        recv = best_model<false>(want, z);
        if (recv >= 0) {
          if (Tk < reb_until && !hard) deferred = true;
          else kind = TRE_RESCUE;
        }
      }
      if (kind == 0 && recv < 0 && slow) {       // rebalance: Eq. 3 over non-idle models
        const unsigned want[2] = {surp_m[0] | nom_m[0] | crit_m[0],
                                  surp_m[1] | nom_m[1] | crit_m[1]};
        recv = best_model<false>(want, z);
        if (recv >= 0 && value(z, recv) < (T)1) {
          kind = TRE_REBALANCE;
          nom_above = true;
        }
      }
      if (deferred) kind = 0;
      if (kind) {
        const T zr = value(z, recv);
        unsigned above[2];
#pragma unroll
        for (int j = 0; j < 2; ++j)
          above[j] = nom_above ? __ballot_sync(kFull, z[j] > zr) : kFull;
        // donor preference: idle models (lowest index), then surplus by Z
        // descending, then nominal by Z descending (with nom_above only above
        // the receiver's Z); never critical, never the receiver, never below
        // the floor, never a donor whose latency guard is breached
        auto pick = [&](const int32_t (&rr)[2]) -> int {
          unsigned can[2];
#pragma unroll
          for (int j = 0; j < 2; ++j)
            can[j] = __ballot_sync(kFull, lane + 32 * j != recv && rr[j] > rmin[j] && !held[j]);
          if (can[0] & idle_m[0]) return __ffs(can[0] & idle_m[0]) - 1;
          if (can[1] & idle_m[1]) return 32 + __ffs(can[1] & idle_m[1]) - 1;
          const unsigned su[2] = {can[0] & surp_m[0], can[1] & surp_m[1]};
          const int d = best_model<true>(su, z);
          if (d >= 0) return d;
          const unsigned no[2] = {can[0] & nom_m[0] & above[0], can[1] & nom_m[1] & above[1]};
          return best_model<true>(no, z);
        };
        auto emit = [&](int donor, int seq) {
          if (lane == 0 && nm < b.moves_cap) {
            tre_move mv;
            mv.window = k;
            mv.recv = (int16_t)recv;
            mv.donor = (int16_t)donor;
            mv.kind = (uint8_t)kind;
            mv.seq = (uint8_t)seq;
            mv.reserved = 0;
            b.moves[(size_t)inst * b.moves_cap + nm] = mv;
          }
          ++nm;
        };
        auto give = [&](int m, int d) {
          if (m == lane) r[0] += d;
          if (m == lane + 32) r[1] += d;
        };
        auto push = [&](int m, long long t) {
          if (lane == 0) {
            srv[(size_t)m * b.hcap + n_srv[m]] = free_at(t);
            n_srv[m] += 1;
          }
          __syncwarp();
        };
        const long long need = count(fp, recv);
        for (int seq = 0; seq < pacing; ++seq) {
          long long gpu_free = Tk;
          if (pool >= need) {                    // idle capacity first
            pool -= need;
            emit(-1, seq);
          } else {
            // dry run: can the eligible donors cover the receiver's footprint?
            int32_t rr[2] = {r[0], r[1]};
            long long f = pool;
            bool ok = true;
            while (f < need) {
              const int d = pick(rr);
              if (d < 0) {
                ok = false;
                break;
              }
              if (d == lane) rr[0] -= 1;
              if (d == lane + 32) rr[1] -= 1;
              f += count(fp, d);
            }
            if (!ok) break;
            // commit: the same releases, each the donor's server that frees first
            f = pool;
            while (f < need) {
              const int d = pick(r);
              give(d, -1);
              f += count(fp, d);
              emit(d, seq);
              uint32_t* sv = srv + (size_t)d * b.hcap;
              const int n = n_srv[d];
              int at;
              const long long fr = Servers{sv, n}.first(at);
              const long long drained = max(fr, Tk);
              __syncwarp();
              if (lane == 0) {
                sv[at] = sv[n - 1];
                n_srv[d] = n - 1;
              }
              __syncwarp();
              gpu_free = max(gpu_free, drained + b.sleep_ms);
            }
            pool = f - need;
          }
          give(recv, 1);
          push(recv, gpu_free + b.wake_ms);
          if (kind == TRE_REBALANCE) reb_until = max(reb_until, gpu_free + (long long)b.wake_ms);
        }
#pragma unroll
        for (int j = 0; j < 2; ++j)
          if (lane + 32 * j < M) rep[lane + 32 * j] = r[j];
      }
    }
    __syncthreads();
  }
  __syncthreads();
  // requests never started count against the SLO with their first token at
  // the end of the grid
  for (int m = wid; m < M; m += n_warps) {
    const ModelState<T>& s = st_m[m];
    unsigned met = 0;
    if (b.slo_ms) {
      for (int q = s.head + lane; q < s.end; q += 32)
        met += (long long)span - (long long)b.grp[2 * (size_t)q].x <= (long long)b.slo_ms[m];
      met = __reduce_add_sync(kFull, met);
    }
    if (lane == 0) {
      if (b.slo_ms && b.slo_met) b.slo_met[(size_t)inst * M + m] = (int64_t)(s.met + met);
      if (b.served) b.served[(size_t)inst * M + m] = (int64_t)(s.head - b.base[m]);
      b.r_final[(size_t)inst * M + m] = rep[m];
    }
  }
  if (threadIdx.x == 0) {
    b.n_moves[inst] = nm;
    if (nm > b.moves_cap) b.diag->err = TRE_EOVERFLOW;
  }
}

// what a block may opt into, less the reserve of the system
constexpr size_t kReplaySmemMax = 224 * 1024;

}  // namespace

template <class T> void replay_ws_layout(Arena& a, ReplayBatch<T>& b, ReplayWs& w) {
  const int M = b.M, K = b.K;
  const size_t n = (size_t)std::max<int64_t>(b.lat.n, 1);
  w.n_blk = (int)((b.lat.n + kGroupBlock - 1) / kGroupBlock);
  w.vm = a.take<int8_t>(n);
  w.arr_cnt = a.take<int32_t>((size_t)K * M + 1);
  w.blk_cnt = a.take<int32_t>((size_t)std::max(w.n_blk, 1) * M);
  w.base = a.take<int32_t>((size_t)M + 1);
  w.acc = a.take<uint32_t>((size_t)b.n_inst * kFarCounts * (K + 1) * M);
  w.grp = a.take<int4>(n * 2);
  auto a16 = [](size_t x) { return (x + 15) & ~(size_t)15; };
  const size_t rows = a16((size_t)M * (sizeof(ModelState<T>) + sizeof(T) + 4 + 4 + 1 + 1));
  const size_t rings = (size_t)kCounts * M * kRing * 4;
  const size_t srv = (size_t)M * b.hcap * 4;
  const bool fits = rows + rings + srv <= kReplaySmemMax;
  b.ring_off = (int)rows;
  b.srv_off = (int)(rows + rings);
  b.smem_bytes = (int)(rows + rings + (fits ? srv : 0));
  b.gsrv = nullptr;
  uint32_t* g = fits ? nullptr : a.take<uint32_t>((size_t)b.n_inst * M * b.hcap);
  b.gsrv = g;
  b.grp = w.grp;
  b.base = w.base;
  b.arr_cnt = w.arr_cnt;
  b.acc = w.acc;
}

template <class T> cudaError_t launch_replay(ReplayBatch<T>& b, ReplayWs& w, cudaStream_t s) {
  const int M = b.M, K = b.K;
  cudaError_t e = cudaMemsetAsync(w.arr_cnt, 0, ((size_t)K * M + 1) * sizeof(int32_t), s);
  if (!e)
    e = cudaMemsetAsync(w.acc, 0, (size_t)b.n_inst * kFarCounts * (K + 1) * M * sizeof(uint32_t), s);
  if (e) return e;
  const FastDiv fwin((uint32_t)b.win);
  if (w.n_blk > 0)
    k_rp_valid<<<w.n_blk, kGroupBlock, 0, s>>>(b.lat, M, fwin, (int64_t)K * b.win, w.vm, w.arr_cnt,
                                               w.blk_cnt);
  k_rp_offsets<<<1, 1024, 0, s>>>(M, w.n_blk, w.blk_cnt, w.base);
  if (w.n_blk > 0)
    k_rp_group<<<w.n_blk, kGroupBlock, 0, s>>>(b.lat, M, w.vm, w.blk_cnt, w.base, w.grp);
  if ((e = cudaGetLastError())) return e;
  if (b.o_ts && b.lat.n > 0) {
    k_rp_init_records<<<(unsigned)device_sm_count() * 8, 256, 0, s>>>(
        b.lat.n, b.n_inst, (int32_t)(K * b.win), w.vm, b.o_ts, b.o_tf, b.o_te);
    if ((e = cudaGetLastError())) return e;
  }
  // two warps a model while their barriers and the block's warps suffice
  const bool pair = M <= kMaxPairs;
  auto f = pair ? k_replay<T, true> : k_replay<T, false>;
  if ((e = func_smem_once((const void*)f, (int)kReplaySmemMax, false))) return e;
  f<<<(unsigned)b.n_inst, pair ? 64 * M : 32 * std::min(M, kMaxWarps), (size_t)b.smem_bytes, s>>>(b);
  return cudaGetLastError();
}

template void replay_ws_layout<float>(Arena&, ReplayBatch<float>&, ReplayWs&);
template void replay_ws_layout<double>(Arena&, ReplayBatch<double>&, ReplayWs&);
template cudaError_t launch_replay<float>(ReplayBatch<float>&, ReplayWs&, cudaStream_t);
template cudaError_t launch_replay<double>(ReplayBatch<double>&, ReplayWs&, cudaStream_t);

}  // namespace tre
