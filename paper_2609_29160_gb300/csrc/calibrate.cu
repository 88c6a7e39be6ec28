// Calibration of the healthy boundary theta (Sec. III-B: the lowest smoothed TSS
// value at which the SLO reliability target is still met), for a batch of
// series at once.
//
// For model m, let the calibration windows be those with at least one arrival,
// not idle, S > 0. For a value s let C(s) be the number of calibration windows
// with S >= s and H(s) the healthy ones among them. theta is the smallest S
// value s with H(s) >= reliability * C(s).
//
// Instead of sorting, each (series, model) packs its (S, healthy) pairs into
// unsigned keys (the bit pattern of a positive float orders like the float)
// and one CTA finds theta from a histogram over the key range: per bucket, in
// parallel, the exact test at its smallest value (everything at or above it
// included) and an upper bound for any value inside it (only its healthy
// windows added). Values of buckets below the lowest one that passes, but whose
// bound does, are tested one by one. When too many would have to be, a descent
// over the key range refines one bucket after another. Counts are exact
// integers and the tests give the definition's double comparison, so theta is
// exact.
#include <cooperative_groups.h>

#include <algorithm>

#include "common.cuh"
#include "internal.h"

namespace tre {
namespace {

constexpr int kThrTable = 4096;
constexpr int kNB = 1024;           // buckets per level = threads per CTA
constexpr int kWarps = kNB / 32;

template <class T> struct KeyOf;
template <> struct KeyOf<float> {
  using U = uint32_t;
  static constexpr int kLevels = 4;   // 31 key bits, >= 10 bits resolved per level
};
template <> struct KeyOf<double> {
  using U = unsigned long long;
  static constexpr int kLevels = 7;   // 63 key bits
};

__device__ __forceinline__ float value_of(uint32_t k) { return __uint_as_float(k); }
__device__ __forceinline__ double value_of(unsigned long long k) {
  return __longlong_as_double((long long)k);
}

// (double)h >= rate * (double)c. Decided in float where the two sides are
// further apart than the float conversions and the product can be off (a few
// 2^-24 of either side); only near ties take the double expression (the FP64
// pipe has two lanes an SM: testing all 4096 buckets in double took 8 us).
__device__ __forceinline__ bool at_least(uint32_t h, uint32_t c, double rate, float rate_f) {
  const float x = (float)h, t = rate_f * (float)c;
  const float margin = 1.f + (x + fabsf(t)) * 0x1p-20f;
  if (x >= t + margin) return true;
  if (x <= t - margin) return false;
  return (double)h >= rate * (double)c;
}

// smallest integer n with (double)n >= ok_frac * (double)a
__device__ __forceinline__ int32_t healthy_from(double ok_frac, int a) {
  const double v = ok_frac * (double)a;
  if (!(v <= 2147483647.0)) return 0x7fffffff;        // unreachable (or NaN)
  if (v <= -2147483647.0) return -0x7fffffff;
  return (int32_t)ceil(v);
}

// thr[a] = smallest integer n with (double)n >= ok_frac * (double)a; also
// resets the per-(series, model) candidate key ranges filled by k_pack
template <class U>
__global__ void k_thr(double ok_frac, int32_t* thr, int n_sm, U* kmin, U* kmax, uint32_t* ncand) {
  const int a = blockIdx.x * blockDim.x + threadIdx.x;
  if (a < n_sm) {
    kmin[a] = ~(U)0;
    kmax[a] = 0;
    ncand[a] = 0;
  }
  if (a >= kThrTable) return;
  thr[a] = healthy_from(ok_frac, a);
}

__device__ __forceinline__ bool healthy(uint32_t n_arr, uint32_t n_met, const int32_t* thr,
                                        double ok_frac) {
  if (n_arr < (uint32_t)kThrTable) return (int64_t)n_met >= (int64_t)thr[n_arr];
  return (double)n_met >= ok_frac * (double)n_arr;
}

// [K][M] S, class, packed SLO counts of every series -> [M][K] packed keys
// (0 = not a calibration window) at the series' element offset, plus each
// (series, model)'s smallest and largest candidate key and candidate count.
// A CTA transposes one tile of TK windows x TM models (TM = the model count
// rounded up to a power of two, at most 32; TK * TM = 1024) through shared
// memory; every thread of a CTA keeps to one model of the tile.
constexpr int kPackThreads = 256;
constexpr int kPackTile = 1024;
struct PackPlan {
  int lg_tm, tm, lg_tk, tk, m_tiles;
  int tile_base[kMaxSeries + 1];   // prefix of tiles per series
};

__device__ __forceinline__ uint32_t warp_min(uint32_t v) { return __reduce_min_sync(0xffffffffu, v); }
__device__ __forceinline__ uint32_t warp_max(uint32_t v) { return __reduce_max_sync(0xffffffffu, v); }
__device__ __forceinline__ unsigned long long warp_min(unsigned long long v) {
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long y = __shfl_xor_sync(0xffffffffu, v, o);
    v = y < v ? y : v;
  }
  return v;
}
__device__ __forceinline__ unsigned long long warp_max(unsigned long long v) {
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long y = __shfl_xor_sync(0xffffffffu, v, o);
    v = y > v ? y : v;
  }
  return v;
}

__device__ __forceinline__ void load4(const float* p, float (&v)[4]) {
  const float4 q = *reinterpret_cast<const float4*>(p);
  v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
}
__device__ __forceinline__ void load4(const double* p, double (&v)[4]) {
  const double2 a = reinterpret_cast<const double2*>(p)[0];
  const double2 b = reinterpret_cast<const double2*>(p)[1];
  v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
}

// The same packing with 16-byte loads, for model counts that fill whole tile
// rows (M a multiple of TM and of 4, 16-byte aligned arrays): a thread reads
// four consecutive models of one window; the candidate range and count of a
// tile row come from warp reductions over the transposed tile.
template <class T>
__global__ void __launch_bounds__(kPackThreads)
k_pack_vec(const __grid_constant__ SeriesTable<T> tab, const __grid_constant__ PackPlan pp,
           const T* __restrict__ S, const uint8_t* __restrict__ cls,
           const unsigned long long* __restrict__ slo, const int32_t* __restrict__ thr,
           double ok_frac, typename KeyOf<T>::U* __restrict__ keys,
           typename KeyOf<T>::U* kmin_g, typename KeyOf<T>::U* kmax_g, uint32_t* ncand_g) {
  using U = typename KeyOf<T>::U;
  static_assert(kPackTile == 4 * kPackThreads, "four elements per thread");
  __shared__ U tile[kPackTile + 32];
  __shared__ U smin[32], smax[32];
  __shared__ uint32_t scnt[32];
  const int s = prefix_index(pp.tile_base, tab.n, blockIdx.x);
  const int M = tab.M, K = tab.K[s];
  const int t_loc = blockIdx.x - pp.tile_base[s];
  const int kt = pp.m_tiles == 1 ? t_loc : t_loc / pp.m_tiles;
  const int k0 = kt * pp.tk, m0 = (t_loc - kt * pp.m_tiles) * pp.tm;
  const size_t off = (size_t)tab.off[s];
  const int tid = threadIdx.x;
  if (tid < 32) {
    smin[tid] = ~(U)0;
    smax[tid] = 0;
    scnt[tid] = 0;
  }
  const int TKp = pp.tk + 1;
  const int e4 = tid * 4;
  const int kk = e4 >> pp.lg_tm, mm = e4 & (pp.tm - 1);
  const int k = k0 + kk;
  U v[4] = {0, 0, 0, 0};
  if (k < K) {
    const size_t x = off + (size_t)k * M + m0 + mm;
    T sv[4];
    load4(S + x, sv);
    const uchar4 c4 = *reinterpret_cast<const uchar4*>(cls + x);
    const ulonglong2 a = reinterpret_cast<const ulonglong2*>(slo + x)[0];
    const ulonglong2 b = reinterpret_cast<const ulonglong2*>(slo + x)[1];
    const unsigned long long cv[4] = {a.x, a.y, b.x, b.y};
    const uint8_t iv[4] = {c4.x, c4.y, c4.z, c4.w};
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const uint32_t n_arr = (uint32_t)cv[u];
      if (iv[u] != kIdle && n_arr >= 1 && sv[u] > (T)0) {
        const bool h = healthy(n_arr, (uint32_t)(cv[u] >> 32), thr, ok_frac);
        v[u] = ((U)key_of(sv[u]) << 1) | (U)(h ? 1 : 0);
      }
    }
  }
#pragma unroll
  for (int u = 0; u < 4; ++u) tile[(mm + u) * TKp + kk] = v[u];
  __syncthreads();
  // tile rows are models: a warp's 32 consecutive elements share one row
#pragma unroll
  for (int j = 0; j < kPackTile / kPackThreads; ++j) {
    const int e = tid + j * kPackThreads;
    const int r = e >> pp.lg_tk, kr = e & (pp.tk - 1);
    const int kg = k0 + kr;
    const U w = tile[r * TKp + kr];
    const bool in = kg < K;
    if (in) keys[off + (size_t)(m0 + r) * K + kg] = w;
    const bool cand = in && w != 0;
    const U lo = warp_min(cand ? (U)(w >> 1) : ~(U)0);
    const U hi = warp_max(cand ? (U)(w >> 1) : (U)0);
    const uint32_t nc = __popc(__ballot_sync(0xffffffffu, cand));
    if ((tid & 31) == 0 && nc) {
      atomicMin(&smin[r], lo);
      atomicMax(&smax[r], hi);
      atomicAdd(&scnt[r], nc);
    }
  }
  __syncthreads();
  if (tid < pp.tm && scnt[tid]) {
    const size_t g = (size_t)s * M + m0 + tid;
    atomicMin(&kmin_g[g], smin[tid]);
    atomicMax(&kmax_g[g], smax[tid]);
    atomicAdd(&ncand_g[g], scnt[tid]);
  }
}

template <class T>
__global__ void __launch_bounds__(kPackThreads)
k_pack(const __grid_constant__ SeriesTable<T> tab, const __grid_constant__ PackPlan pp,
       const T* __restrict__ S, const uint8_t* __restrict__ cls,
       const unsigned long long* __restrict__ slo, const int32_t* __restrict__ thr,
       double ok_frac, typename KeyOf<T>::U* __restrict__ keys, typename KeyOf<T>::U* kmin_g,
       typename KeyOf<T>::U* kmax_g, uint32_t* ncand_g) {
  using U = typename KeyOf<T>::U;
  __shared__ U tile[kPackTile + 32];
  __shared__ U smin[32], smax[32];
  __shared__ uint32_t scnt[32];
  const int s = prefix_index(pp.tile_base, tab.n, blockIdx.x);
  const int M = tab.M, K = tab.K[s];
  const int t_loc = blockIdx.x - pp.tile_base[s];
  const int kt = pp.m_tiles == 1 ? t_loc : t_loc / pp.m_tiles;
  const int k0 = kt * pp.tk, m0 = (t_loc - kt * pp.m_tiles) * pp.tm;
  const size_t off = (size_t)tab.off[s];
  const int tid = threadIdx.x;
  const int mm = tid & (pp.tm - 1);
  const int m = m0 + mm;
  if (tid < 32) {
    smin[tid] = ~(U)0;
    smax[tid] = 0;
    scnt[tid] = 0;
  }
  U lmin = ~(U)0, lmax = 0;
  uint32_t lc = 0;
  const int TKp = pp.tk + 1;   // padded row of the transposed tile
  constexpr int J = kPackTile / kPackThreads;
  // every load of the thread's elements first, then the threshold lookups,
  // then the keys: more requests in flight per thread
  unsigned long long cj[J];
  T sj[J];
  uint8_t ij[J];
  bool in[J];
#pragma unroll
  for (int j = 0; j < J; ++j) {
    const int k = k0 + ((tid + j * kPackThreads) >> pp.lg_tm);
    in[j] = k < K && m < M;
    const size_t x = off + (size_t)k * M + m;
    cj[j] = in[j] ? slo[x] : 0ull;
    sj[j] = in[j] ? S[x] : (T)0;
    ij[j] = in[j] ? cls[x] : kIdle;
  }
  bool hj[J];
#pragma unroll
  for (int j = 0; j < J; ++j) hj[j] = healthy((uint32_t)cj[j], (uint32_t)(cj[j] >> 32), thr, ok_frac);
#pragma unroll
  for (int j = 0; j < J; ++j) {
    const int kk = (tid + j * kPackThreads) >> pp.lg_tm;
    U v = 0;
    if (in[j] && ij[j] != kIdle && (uint32_t)cj[j] >= 1 && sj[j] > (T)0) {
      const U key = (U)key_of(sj[j]);
      v = (key << 1) | (U)(hj[j] ? 1 : 0);
      lmin = key < lmin ? key : lmin;
      lmax = key > lmax ? key : lmax;
      ++lc;
    }
    tile[mm * TKp + kk] = v;
  }
  __syncthreads();
  if (lc) {
    atomicMin(&smin[mm], lmin);
    atomicMax(&smax[mm], lmax);
    atomicAdd(&scnt[mm], lc);
  }
#pragma unroll
  for (int j = 0; j < kPackTile / kPackThreads; ++j) {
    const int e = tid + j * kPackThreads;
    const int r = e >> pp.lg_tk, kk = e & (pp.tk - 1);
    const int mo = m0 + r, k = k0 + kk;
    if (mo < M && k < K) keys[off + (size_t)mo * K + k] = tile[r * TKp + kk];
  }
  __syncthreads();
  if (tid < pp.tm && m0 + tid < M && scnt[tid]) {
    const size_t g = (size_t)s * M + m0 + tid;
    atomicMin(&kmin_g[g], smin[tid]);
    atomicMax(&kmax_g[g], smax[tid]);
    atomicAdd(&ncand_g[g], scnt[tid]);
  }
}

// exclusive suffix sums of two values over the block (sums over threads > tid)
__device__ __forceinline__ int2 block_suffix(int a, int b, int2* red) {
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31, wid = threadIdx.x / 32;
  int ia = a, ib = b;               // inclusive suffix within the warp
  for (int o = 1; o < 32; o <<= 1) {
    const int xa = __shfl_down_sync(full, ia, o), xb = __shfl_down_sync(full, ib, o);
    if (lane + o < 32) {
      ia += xa;
      ib += xb;
    }
  }
  if (lane == 0) red[wid] = make_int2(ia, ib);
  __syncthreads();
  const int2 w = red[lane];
  const int above_a = __reduce_add_sync(full, lane > wid ? w.x : 0);
  const int above_b = __reduce_add_sync(full, lane > wid ? w.y : 0);
  __syncthreads();
  return make_int2(ia - a + above_a, ib - b + above_b);
}

__device__ __forceinline__ int block_min(int v, int* red) {
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31, wid = threadIdx.x / 32;
  v = __reduce_min_sync(full, v);
  if (lane == 0) red[wid] = v;
  __syncthreads();
  v = __reduce_min_sync(full, red[lane]);
  __syncthreads();
  return v;
}
static_assert(kWarps == 32, "one block-wide value per lane");

constexpr int kFine = 4096;     // buckets of the first histogram
constexpr int kUnroll = 8;      // keys per thread whose loads are issued together
constexpr int kCap = 2048;      // most keys the exact pass tests one by one
constexpr int kDirectK = kUnroll * kNB;       // longest series searched without packing
constexpr int64_t kDirectCells = 1 << 18;     // and largest table: a CTA reads one column of
                                              // the rows, 4 to 8 bytes of each 32-byte sector

template <class T> size_t search_smem_bytes() {
  using U = typename KeyOf<T>::U;
  const size_t fast = (size_t)kFine * (5 * 4) + (size_t)kCap * sizeof(U);
  const size_t descent = (size_t)KeyOf<T>::kLevels * kNB * (4 + 4 + sizeof(U));
  return fast > descent ? fast : descent;
}

// One CTA per (series, model), or a cluster of CL of them. DIRECT: the keys are made
// here, from the model's column of S, classes and counts, and stay in registers (series of up
// to kDirectK windows): one launch where packing, its threshold table and the
// search were three. Otherwise they come from the packing pass, and are read
// again for the gather. What bounds a search is its chain of block-wide steps.
// 8 models, 3,600 windows: 12.0 us in one launch (25.3 in three, with a bitonic
// sort of the gathered keys and every test in double; 14.0 with 4,096 buckets, four
// a thread, where a short series fills a bucket a thread as well); 16 models, 43,200
// windows: 21.6 us (30.5); the sweep's 224 searches: 24.5 us (33.3).
//
// With CL CTAs each reads its part of the keys: they count into their own
// histograms, the first adds them up and chooses the buckets, all list the keys
// of those buckets in the first one's memory, and the first tests them. Long
// series leave SMs idle otherwise: 64 series of 864,000 windows took 250 us.
template <class T, bool DIRECT, int CL>
__global__ void __launch_bounds__(kNB, !DIRECT && sizeof(T) == 4 ? 2 : 1)
k_search(const __grid_constant__ SeriesTable<T> tab, typename KeyOf<T>::U* __restrict__ keys,
         const typename KeyOf<T>::U* kmin_g, const typename KeyOf<T>::U* kmax_g,
         const uint32_t* ncand_g, const T* __restrict__ S, const uint8_t* __restrict__ cls,
         const unsigned long long* __restrict__ slo, double ok_frac, double reliability, T* theta,
         T* theta1, tre_diag* diag) {
  using U = typename KeyOf<T>::U;
  constexpr int NL = KeyOf<T>::kLevels;
  constexpr int kFineHere = DIRECT ? kNB : kFine;   // a bucket a thread on short series
  constexpr int kThrDirect = 256;
  extern __shared__ __align__(16) unsigned char dyn[];
  __shared__ U lo_s[NL], hi_s[NL];
  __shared__ int shift_s[NL], pos_s[NL];
  __shared__ int cab_s[NL], hab_s[NL];
  __shared__ int2 red2[kWarps];
  __shared__ int red32[kWarps];
  __shared__ U redU[2][kWarps];
  __shared__ int thr_s[kThrDirect];
  __shared__ U bfmin_s, best_s;
  __shared__ int plan_s[2];       // keys listed, lowest found bucket
  namespace cg = cooperative_groups;
  static_assert(!DIRECT || CL == 1, "short series need one CTA");
  const int M = tab.M;
  const int sm = blockIdx.x / CL, rank = blockIdx.x % CL;
  const int s = sm / M, m = sm % M;
  const int K = tab.K[s];
  const int part = (K + CL - 1) / CL, i_lo = rank * part, i_hi = min(K, i_lo + part);
  U* mk = keys + (size_t)tab.off[s] + (size_t)m * K;
  const int tid = threadIdx.x, lane = tid & 31;
  const size_t out = (size_t)s * M + m;
  T* const th_out = theta1 && s == 1 ? theta1 + m : theta + out;
  const float rel_f = (float)reliability;
  int32_t* fcnt = reinterpret_cast<int32_t*>(dyn);
  int32_t* fhl = fcnt + kFineHere;
  int32_t* fst = fhl + kFineHere;                   // where a selected bucket's keys start, -1 if not
  int32_t* fca = fst + kFineHere;                   // windows in buckets above
  int32_t* fha = fca + kFineHere;                   // healthy windows in buckets above
  U* list = reinterpret_cast<U*>(fha + kFineHere);
  for (int b = tid; b < kFineHere; b += kNB) {
    fcnt[b] = 0;
    fhl[b] = 0;
  }
  if (tid == 0) {
    bfmin_s = ~(U)0;
    best_s = ~(U)0;
  }

  // ---- candidate keys: their range and number -------------------------------
  U pv[kUnroll];
  U kmin, kmax;
  uint32_t ncand;
  if (DIRECT) {
    if (tid < kThrDirect) thr_s[tid] = healthy_from(ok_frac, tid);
    T sv[kUnroll];
    uint8_t iv[kUnroll];
    unsigned long long cv[kUnroll];
#pragma unroll
    for (int u = 0; u < kUnroll; ++u) {
      const int k = u * kNB + tid;
      const size_t x = (size_t)tab.off[s] + (size_t)k * M + m;
      const bool in = k < K;
      sv[u] = in ? S[x] : (T)0;
      iv[u] = in ? cls[x] : kIdle;
      cv[u] = in ? slo[x] : 0ull;
    }
    __syncthreads();
    const float ok_f = (float)ok_frac;
    U lo = ~(U)0, hi = 0;
    int n = 0;
#pragma unroll
    for (int u = 0; u < kUnroll; ++u) {
      const uint32_t n_arr = (uint32_t)cv[u], n_met = (uint32_t)(cv[u] >> 32);
      pv[u] = 0;
      if (iv[u] != kIdle && n_arr >= 1 && sv[u] > (T)0) {
        const bool h = n_arr < (uint32_t)kThrDirect ? (int64_t)n_met >= (int64_t)thr_s[n_arr]
                                                    : at_least(n_met, n_arr, ok_frac, ok_f);
        const U key = (U)key_of(sv[u]);
        pv[u] = (key << 1) | (U)(h ? 1 : 0);
        lo = key < lo ? key : lo;
        hi = key > hi ? key : hi;
        ++n;
      }
    }
    lo = warp_min(lo);
    hi = warp_max(hi);
    n = __reduce_add_sync(0xffffffffu, n);
    if (lane == 0) {
      redU[0][tid / 32] = lo;
      redU[1][tid / 32] = hi;
      red32[tid / 32] = n;
    }
    __syncthreads();
    kmin = warp_min(redU[0][lane]);
    kmax = warp_max(redU[1][lane]);
    ncand = (uint32_t)__reduce_add_sync(0xffffffffu, red32[lane]);
  } else {
    ncand = ncand_g[out];
    kmin = kmin_g[out];
    kmax = kmax_g[out];
  }
  if (ncand == 0) {
    if (tid == 0 && rank == 0) {
      *th_out = (T)1;
      atomicAdd(&diag->degenerate_calib, 1ull);
    }
    return;
  }

  // ---- fast path -----------------------------------------------------------
  // A fine histogram over [kmin, kmax]; per bucket the exact test at its
  // smallest value ("found") and the bound for values inside it ("maybe").
  // With bf the lowest found bucket, theta is either a value inside a maybe
  // bucket below bf or the smallest value of bf. Those maybe buckets' keys are
  // gathered bucket by bucket, and each is tested with the counts of the keys
  // not below it in its own bucket: no order within a bucket is needed.
  {
    int sh = 0;
    while (sh < 63 && ((kmax - kmin) >> sh) >= (U)kFineHere) ++sh;
    __syncthreads();
    // with fewer than 2^16 candidates, a bucket's count and healthy count
    // share one 32-bit word (one atomic per key)
    const bool packed = ncand < 65536u;
    uint32_t* fpk = reinterpret_cast<uint32_t*>(fcnt);
    auto each_key = [&](auto&& f) {
      if (DIRECT) {
#pragma unroll
        for (int u = 0; u < kUnroll; ++u)
          if (pv[u]) f(pv[u], (int)(((pv[u] >> 1) - kmin) >> sh));
      } else {
        for (int i0 = i_lo; i0 < i_hi; i0 += kNB * kUnroll) {
#pragma unroll
          for (int u = 0; u < kUnroll; ++u) {
            const int i = i0 + u * kNB + tid;
            pv[u] = i < i_hi ? mk[i] : (U)0;
          }
#pragma unroll
          for (int u = 0; u < kUnroll; ++u)
            if (pv[u]) f(pv[u], (int)(((pv[u] >> 1) - kmin) >> sh));
        }
      }
    };
    each_key([&](U p, int b) {
      if (packed) {
        atomicAdd(&fpk[b], 1u + ((uint32_t)(p & 1) << 16));
      } else {
        atomicAdd(&fcnt[b], 1);
        if (p & 1) atomicAdd(&fhl[b], 1);
      }
    });
    __syncthreads();
    if constexpr (CL > 1) cg::this_cluster().sync();
    constexpr int PER = kFineHere / kNB;            // consecutive buckets per thread
    int bf = 0x7fffffff, nsel = 0;
    if (rank == 0) {
    const int b0 = tid * PER;
    int cb[PER], hb[PER], tc = 0, th = 0;
#pragma unroll
    for (int j = 0; j < PER; ++j) {
      const uint32_t v = fpk[b0 + j];
      cb[j] = packed ? (int)(v & 0xffffu) : (int)v;
      hb[j] = packed ? (int)(v >> 16) : fhl[b0 + j];
      if constexpr (CL > 1) {
        // packed sums stay packed: fewer than 2^16 candidates in all
        const cg::cluster_group cl = cg::this_cluster();
#pragma unroll
        for (int r = 1; r < CL; ++r) {
          const uint32_t w = cl.map_shared_rank(fpk, r)[b0 + j];
          cb[j] += packed ? (int)(w & 0xffffu) : (int)w;
          hb[j] += packed ? (int)(w >> 16) : cl.map_shared_rank(fhl, r)[b0 + j];
        }
      }
      tc += cb[j];
      th += hb[j];
    }
    const int2 above = block_suffix(tc, th, red2);
    int ca[PER], ha[PER], my_found = 0x7fffffff;
    uint32_t maybe_bits = 0;
    {
      int c = above.x, h = above.y;
#pragma unroll
      for (int j = PER - 1; j >= 0; --j) {
        ca[j] = c;
        ha[j] = h;
        if (cb[j] > 0) {
          if (at_least(h + hb[j], c + cb[j], reliability, rel_f)) {
            my_found = b0 + j;
          } else if (at_least(h + hb[j] + 1, c + hb[j], reliability, rel_f)) {
            // a value inside adds at most the bucket's healthy windows to those
            // above; one window of slack keeps the bound valid under rounding
            maybe_bits |= 1u << j;
          }
        }
        c += cb[j];
        h += hb[j];
      }
    }
    bf = block_min(my_found, red32);
    int my_sel = 0;
#pragma unroll
    for (int j = 0; j < PER; ++j) {
      if (b0 + j >= bf) maybe_bits &= ~(1u << j);
      my_sel += maybe_bits >> j & 1u ? cb[j] : 0;
    }
    const int sel_above = block_suffix(my_sel, 0, red2).x;
    if (tid == 0) red32[0] = sel_above + my_sel;
    __syncthreads();
    nsel = red32[0];
    if (nsel <= kCap) {
      int run = sel_above;
#pragma unroll
      for (int j = 0; j < PER; ++j) {
        const bool on = maybe_bits >> j & 1u;
        fst[b0 + j] = on ? run : -1;
        fca[b0 + j] = ca[j];
        fha[b0 + j] = ha[j];
        fcnt[b0 + j] = cb[j];
        fhl[b0 + j] = 0;                        // from here on: keys of the bucket listed
        run += on ? cb[j] : 0;
      }
    }
    if (tid == 0) {
      plan_s[0] = nsel;
      plan_s[1] = bf;
    }
    }
    // where the buckets' keys go: this CTA's copy of the table, the first one's list
    int32_t* place = fhl;
    U* keep = list;
    if constexpr (CL > 1) {
      const cg::cluster_group cl = cg::this_cluster();
      cl.sync();
      if (rank > 0) {
        const int32_t* src = cl.map_shared_rank(fst, 0);
        for (int q = tid; q < kFineHere; q += kNB) fst[q] = src[q];
        nsel = cl.map_shared_rank(plan_s, 0)[0];
        bf = cl.map_shared_rank(plan_s, 0)[1];
      }
      // every CTA, the first one too, adds to the places by cluster addresses: the
      // same 32-bit addition from all of them
      place = cl.map_shared_rank(fhl, 0);
      keep = cl.map_shared_rank(list, 0);
      cl.sync();                    // the first CTA may end from here on unless keys are listed
    }
    __syncthreads();
    if (nsel <= kCap) {
      if (nsel > 0 || bf != 0x7fffffff) {
        U lmin = ~(U)0;
        each_key([&](U p, int b) {
          const int st = fst[b];
          if (st >= 0) keep[st + atomicAdd(&place[b], 1)] = p;
          if (b == bf && (p >> 1) < lmin) lmin = p >> 1;
        });
        if (lmin != ~(U)0) atomicMin(&bfmin_s, lmin);
        if constexpr (CL > 1) {
          // each CTA's smallest is its own until all have it. (With one minimum in the
          // first CTA's memory, its own by shared and the others' by cluster addresses,
          // boundaries in double were one value off now and then; that the two do not
          // exclude each other in 64 bits is inferred from this, not documented.)
          const cg::cluster_group cl = cg::this_cluster();
          cl.sync();
          if (rank == 0 && tid == 0)
            for (int r = 1; r < CL; ++r) {
              const U v = *cl.map_shared_rank(&bfmin_s, r);
              if (v < bfmin_s) bfmin_s = v;
            }
          cl.sync();
          if (rank > 0) return;
        }
        __syncthreads();
        U best = ~(U)0;
        for (int i = tid; i < nsel; i += kNB) {
          const U key = list[i] >> 1;
          const int b = (int)((key - kmin) >> sh);
          const int st = fst[b], e = st + fcnt[b];
          int C = fca[b], H = fha[b];
          for (int j = st; j < e; ++j) {
            const U o = list[j];
            const bool ge = (o >> 1) >= key;
            C += ge;
            H += ge && (o & 1);
          }
          if (key < best && at_least(H, C, reliability, rel_f)) best = key;
        }
        if (best != ~(U)0) atomicMin(&best_s, best);
        __syncthreads();
      }
      if (rank > 0) return;
      if (tid == 0) {
        if (best_s != ~(U)0) {
          *th_out = value_of(best_s);
        } else if (bf != 0x7fffffff) {
          *th_out = value_of(bfmin_s);
        } else {
          *th_out = value_of(kmax);
          atomicAdd(&diag->degenerate_calib, 1ull);
        }
      }
      return;
    }
  }
  if (rank > 0) return;             // the first CTA refines alone
  if (DIRECT) {
    // the descent reads the keys from memory
#pragma unroll
    for (int u = 0; u < kUnroll; ++u)
      if (u * kNB + tid < K) mk[u * kNB + tid] = pv[u];
  }
  __syncthreads();

  // ---- fallback: radix descent over the key range (many candidate keys) ----
  int32_t (*cnt)[kNB] = reinterpret_cast<int32_t (*)[kNB]>(dyn);
  int32_t (*hl)[kNB] = reinterpret_cast<int32_t (*)[kNB]>(dyn + (size_t)NL * kNB * 4);
  U (*mn)[kNB] = reinterpret_cast<U (*)[kNB]>(dyn + (size_t)NL * kNB * 8);
  auto build = [&](int l) {
    cnt[l][tid] = 0;
    hl[l][tid] = 0;
    mn[l][tid] = ~(U)0;
    __syncthreads();
    const U lo = lo_s[l], hi = hi_s[l];
    const int sh = shift_s[l];
    for (int i0 = 0; i0 < K; i0 += kNB) {
      const int i = i0 + tid;
      const U p = i < K ? mk[i] : (U)0;
      const U key = p >> 1;
      const bool in = p != 0 && key >= lo && key <= hi;
      const int b = in ? (int)((key - lo) >> sh) : -1;
      const unsigned act = __ballot_sync(0xffffffffu, in);
      if (in) {
        const unsigned grp = __match_any_sync(act, b);
        const unsigned hgrp = __ballot_sync(grp, (p & 1) != 0);
        if (lane == __ffs(grp) - 1) {
          atomicAdd(&cnt[l][b], __popc(grp));
          if (hgrp) atomicAdd(&hl[l][b], __popc(hgrp));
        }
        if (key < mn[l][b]) atomicMin(&mn[l][b], key);
      }
    }
    __syncthreads();
  };
  auto set_range = [&](int l, U lo, U hi, int ca, int ha) {
    int sh = 0;
    while (sh < 63 && ((hi - lo) >> sh) >= (U)kNB) ++sh;
    lo_s[l] = lo;
    hi_s[l] = hi;
    shift_s[l] = sh;
    pos_s[l] = 0;
    cab_s[l] = ca;
    hab_s[l] = ha;
  };
  if (tid == 0) set_range(0, kmin, kmax, 0, 0);
  __syncthreads();
  build(0);
  int l = 0;
  while (true) {
    const int2 up = block_suffix(cnt[l][tid], hl[l][tid], red2);
    const int c_above = up.x + cab_s[l], h_above = up.y + hab_s[l];
    const int32_t c = cnt[l][tid], h = hl[l][tid];
    int cand = 0x7fffffff;
    int kind = 0;   // 1 = its smallest value qualifies, 2 = may contain one
    if (c > 0 && tid >= pos_s[l]) {
      if ((double)(h_above + h) >= reliability * (double)(c_above + c)) {
        kind = 1;
      } else if (shift_s[l] > 0 &&
                 (double)(h_above + h + 1) >= reliability * (double)(c_above + h)) {
        kind = 2;
      }
      if (kind) cand = tid;
    }
    const int b = block_min(cand, red32);
    if (b == 0x7fffffff) {
      if (l == 0) {
        if (tid == 0) {
          *th_out = value_of(kmax);
          atomicAdd(&diag->degenerate_calib, 1ull);
        }
        return;
      }
      --l;
      __syncthreads();
      continue;
    }
    if (tid == b) red32[0] = kind;
    __syncthreads();
    const int kb = red32[0];
    if (kb == 1) {
      if (tid == 0) *th_out = value_of(mn[l][b]);
      return;
    }
    if (tid == b) {
      const U lo = lo_s[l] + ((U)b << shift_s[l]);
      const U hi = lo + (((U)1 << shift_s[l]) - 1);
      pos_s[l] = b + 1;
      set_range(l + 1, lo, hi, c_above, h_above);
    }
    __syncthreads();
    ++l;
    build(l);
  }
}

}  // namespace

template <class T> void calib_ws_layout(Arena& a, int64_t elems, int n_sm, CalibWs<T>& w) {
  using U = typename KeyOf<T>::U;
  w.keys = a.take<U>((size_t)std::max<int64_t>(elems, 1));
  w.thr = a.take<int32_t>(kThrTable);
  const size_t n = (size_t)std::max(n_sm, 1);
  w.kmin = a.take<U>(n);
  w.kmax = a.take<U>(n);
  w.ncand = a.take<uint32_t>(n);
  w.n_sm = n_sm;
}

// series short enough, and a table small enough, to be searched without packing
template <class T> static bool direct_search(const SeriesTable<T>& tab) {
  int64_t cells = 0;
  for (int i = 0; i < tab.n; ++i) {
    if (tab.K[i] > kDirectK) return false;
    cells += (int64_t)tab.K[i] * tab.M;
  }
  return cells <= kDirectCells;
}

// thresholds, packing and search, or the search alone
template <class T> int calibrate_launches(const SeriesTable<T>& tab) {
  return direct_search(tab) ? 1 : 3;
}

template <class T>
cudaError_t launch_calibrate(const SeriesTable<T>& tab, const T* S, const uint8_t* cls,
                             const unsigned long long* slo, double ok_frac, double reliability,
                             T* theta, CalibWs<T>& w, tre_diag* diag, cudaStream_t s, T* theta1) {
  using U = typename KeyOf<T>::U;
  const int n_sm = tab.n * tab.M;
  if (n_sm > w.n_sm) return cudaErrorInvalidValue;
  U* kmin = static_cast<U*>(w.kmin);
  U* kmax = static_cast<U*>(w.kmax);
  const size_t smem = search_smem_bytes<T>();
  if (direct_search(tab)) {
    cudaError_t e = func_smem_once((const void*)k_search<T, true, 1>, (int)smem, true);
    if (e) return e;
    k_search<T, true, 1><<<n_sm, kNB, smem, s>>>(tab, static_cast<U*>(w.keys), kmin, kmax, w.ncand, S,
                                              cls, slo, ok_frac, reliability, theta, theta1, diag);
    return cudaGetLastError();
  }
  const int thr_n = std::max(kThrTable, n_sm);
  k_thr<U><<<(thr_n + 255) / 256, 256, 0, s>>>(ok_frac, w.thr, n_sm, kmin, kmax, w.ncand);
  PackPlan pp;
  pp.lg_tm = 0;
  while ((1 << pp.lg_tm) < tab.M && pp.lg_tm < 5) ++pp.lg_tm;
  pp.tm = 1 << pp.lg_tm;
  pp.lg_tk = 10 - pp.lg_tm;
  pp.tk = 1 << pp.lg_tk;
  static_assert(kPackTile == 1024, "tile of 2^10 elements");
  pp.m_tiles = (tab.M + pp.tm - 1) / pp.tm;
  int tiles = 0;
  for (int i = 0; i < tab.n; ++i) {
    pp.tile_base[i] = tiles;
    tiles += (tab.K[i] + pp.tk - 1) / pp.tk * pp.m_tiles;
  }
  pp.tile_base[tab.n] = tiles;
  const bool vec = tab.M % pp.tm == 0 && tab.M % 4 == 0 &&
                   (((uintptr_t)S | (uintptr_t)cls | (uintptr_t)slo) & 15) == 0;
  if (tiles > 0 && vec)
    k_pack_vec<T><<<tiles, kPackThreads, 0, s>>>(tab, pp, S, cls, slo, w.thr, ok_frac,
                                                 static_cast<U*>(w.keys), kmin, kmax, w.ncand);
  else if (tiles > 0)
    k_pack<T><<<tiles, kPackThreads, 0, s>>>(tab, pp, S, cls, slo, w.thr, ok_frac,
                                             static_cast<U*>(w.keys), kmin, kmax, w.ncand);
  // clusters while the searches leave SMs idle (two share an SM where their
  // tables fit) and a CTA's part still has eight windows a thread
  int cl = 1;
  int64_t longest = 0;
  for (int i = 0; i < tab.n; ++i) longest = std::max<int64_t>(longest, tab.K[i]);
  while (cl < 4 && n_sm * cl * 2 <= 2 * device_sm_count() && longest >= (int64_t)cl * 2 * kDirectK)
    cl *= 2;
  auto search = cl == 4 ? k_search<T, false, 4> : cl == 2 ? k_search<T, false, 2>
                                                          : k_search<T, false, 1>;
  cudaError_t e = func_smem_once((const void*)search, (int)smem, true);
  if (e) return e;
  cudaLaunchConfig_t c = {};
  c.gridDim = dim3((unsigned)(n_sm * cl));
  c.blockDim = dim3(kNB);
  c.dynamicSmemBytes = smem;
  c.stream = s;
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = (unsigned)cl;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  c.attrs = &at;
  c.numAttrs = cl > 1 ? 1 : 0;
  e = cudaLaunchKernelEx(&c, search, tab, static_cast<U*>(w.keys), static_cast<const U*>(kmin),
                         static_cast<const U*>(kmax), static_cast<const uint32_t*>(w.ncand), S,
                         cls, slo, ok_frac, reliability, theta, theta1, diag);
  if (e) return e;
  return cudaGetLastError();
}

template int calibrate_launches<float>(const SeriesTable<float>&);
template int calibrate_launches<double>(const SeriesTable<double>&);
template void calib_ws_layout<float>(Arena&, int64_t, int, CalibWs<float>&);
template void calib_ws_layout<double>(Arena&, int64_t, int, CalibWs<double>&);
template cudaError_t launch_calibrate<float>(const SeriesTable<float>&, const float*,
                                             const uint8_t*, const unsigned long long*, double,
                                             double, float*, CalibWs<float>&, tre_diag*,
                                             cudaStream_t, float*);
template cudaError_t launch_calibrate<double>(const SeriesTable<double>&, const double*,
                                              const uint8_t*, const unsigned long long*, double,
                                              double, double*, CalibWs<double>&, tre_diag*,
                                              cudaStream_t, double*);

}  // namespace tre
