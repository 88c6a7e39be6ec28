// Raw TSS (Eq. 1), exponential smoothing (Sec. III-B), Z = TSS / theta (Eq. 2),
// regions, and the per-window Eq. 3 receiver -- for a batch of series at once.
//
// Eq. 1 is evaluated for every (window, model) in one fully parallel pass. The
// smoothing S_k = alpha*raw_k + (1-alpha)*S_{k-1} is a sequential chain per
// model; to spread it over the GPU and still return exactly the values of the
// sequential definition (one rounding per operation, in order):
//   1. the windows of each series are cut into chunks; one thread per (chunk,
//      model) first runs the recurrence over the B windows before its chunk
//      ("burn-in", started as if the series began there; B ~ c / -ln(1-alpha),
//      so a start error shrinks by e^-c before the chunk: c = 28 for float, 45
//      for double), records the state
//      it reached, then runs its chunk from that state and stores the result;
//   2. one CTA per (series, model) checks the chunk boundaries: a chunk whose
//      recorded burn-in state equals its predecessor's end state (bit for bit,
//      with the same started/not-started flag) goes on where the one before it
//      ends, because every step depends only on the previous state; any other
//      chunk is run again from that end until its new trajectory meets the stored
//      one, in passes over all chunks and in order where passes would be many. A
//      chunk whose burn-in reaches window 0 starts from the true initial state
//      and is exact by construction.
// Where every boundary agrees, the result is the sequential one; chunks are re-run
// only when a burn-in did not converge (idle windows, a tiny alpha), counted in
// tre_diag.ema_resolved.
#include <algorithm>
#include <initializer_list>

#include "common.cuh"
#include "internal.h"

namespace tre {
namespace {

constexpr int kBatch = 16;  // windows loaded ahead in the sequential chains

template <class T> __device__ __forceinline__ T sub_rn(T a, T b);
template <> __device__ __forceinline__ float sub_rn<float>(float a, float b) { return __fsub_rn(a, b); }
template <> __device__ __forceinline__ double sub_rn<double>(double a, double b) { return __dsub_rn(a, b); }

__device__ __forceinline__ bool same_bits(float a, float b) {
  return __float_as_uint(a) == __float_as_uint(b);
}
__device__ __forceinline__ bool same_bits(double a, double b) {
  return __double_as_longlong(a) == __double_as_longlong(b);
}

struct Counts {
  const int32_t *P, *D, *A, *W;
  const int64_t *A_ms, *W_ms;   // time-averaged occupancy (request-ms per window) or null
};

template <class T> __device__ __forceinline__ T from_i64(long long v);
template <> __device__ __forceinline__ float from_i64<float>(long long v) { return __ll2float_rn(v); }
template <> __device__ __forceinline__ double from_i64<double>(long long v) {
  return __ll2double_rn(v);
}

// series of a global segment index (the table has at most 64 entries)
template <class T> __device__ __forceinline__ int series_of_seg(const SeriesTable<T>& t, int seg) {
  return prefix_index(t.seg_base, t.n, seg);
}

template <class T> struct ModelParams {
  T a, b;
};

template <class T>
__device__ __forceinline__ ModelParams<T> load_params(const SeriesTable<T>& t, int s, int m,
                                                      const T* alpha) {
  ModelParams<T> p;
  p.a = alpha ? alpha[m] : t.alpha[s];
  p.b = sub_rn<T>((T)1, p.a);
  return p;
}

// Eq. 1 values of idle windows carry this NaN pattern (arithmetic on the GPU
// only produces the canonical NaN), so the smoothing pass reads one array.
__device__ __forceinline__ float idle_raw(float) { return __uint_as_float(0xffc0deadu); }
__device__ __forceinline__ double idle_raw(double) {
  return __longlong_as_double((long long)0xfff8deaddeadbeefull);
}
__device__ __forceinline__ bool is_idle_raw(float r) { return __float_as_uint(r) == 0xffc0deadu; }
__device__ __forceinline__ bool is_idle_raw(double r) {
  return (unsigned long long)__double_as_longlong(r) == 0xfff8deaddeadbeefull;
}

// ---- pass 0: Eq. 1 for every (window, model) of every series ---------------
// Element-wise passes run over tiles of consecutive elements of one series. On
// large tables a thread takes four consecutive elements, with 16-byte loads and
// stores when they are aligned (scalar ones otherwise), so that enough bytes
// are in flight to cover memory latency. Below kSmallCells a thread takes one
// element and a CTA has four warps, one per scheduler: the divisions of an
// element are its latency (64 cycles an operation in double), and a small table
// leaves the SMs idle anyway (3 models, 600 windows in double: Eq. 1 14.3 us on
// two CTAs).
constexpr int kEwThreads = 256;
constexpr int kSmallThreads = 128;
constexpr int64_t kSmallCells = 1 << 18;
struct TilePlan {
  int tile_base[kMaxSeries + 1];   // prefix of tiles per series
};

// a / b for a divisor above zero and a numerator that often is zero (a window
// without prompt or without decode tokens): the division of a zero leaves the
// short instruction sequence for a subroutine, and takes its whole warp along
// (188 instructions a cell, now 85; Eq. 1 of 64 models, 864,000 windows 299 us,
// now 180), so it divides a one instead and returns the numerator, as 0 / b is.
// The tests on doubles are made on their bits: comparisons of doubles go through
// the pipe that the division itself waits for.
__device__ __forceinline__ bool zero_by_positive(float a, float b) {
  return (a == 0.f) & (b > 0.f);
}
__device__ __forceinline__ bool zero_by_positive(double a, double b) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(a);
  const unsigned long long v = (unsigned long long)__double_as_longlong(b);
  return (u << 1 == 0) & (v - 1 < 0x7ff0000000000000ull);      // 0 < b <= infinity
}
template <class T> __device__ __forceinline__ T div_zero_rn(T a, T b) {
  const bool zero = zero_by_positive(a, b);
  const T q = div_rn(zero ? (T)1 : a, b);
  return zero ? a : q;
}

template <class T>
__device__ __forceinline__ T raw_tss(int32_t p, int32_t d, int32_t a, int32_t w, T dt, T wp,
                                     T wq) {
  const T r_pre = div_zero_rn(from_i32<T>(p), dt);
  const T r_dec = div_zero_rn(from_i32<T>(d), dt);
  const T num = add_rn(mul_rn(wp, r_pre), r_dec);
  T den = add_rn(from_i32<T>(a), mul_rn(wq, from_i32<T>(w)));
  if (den < (T)1) den = (T)1;                       // demand floor of one request
  return div_zero_rn(num, den);
}

// Eq. 1 with the window means of the running and waiting counts: the
// request-milliseconds inside the window divided by its length
template <class T>
__device__ __forceinline__ T raw_tss_mean(int32_t p, int32_t d, long long a_ms, long long w_ms,
                                          T dt, T win, T wp, T wq) {
  const T r_pre = div_zero_rn(from_i32<T>(p), dt);
  const T r_dec = div_zero_rn(from_i32<T>(d), dt);
  const T num = add_rn(mul_rn(wp, r_pre), r_dec);
  const T a = div_zero_rn(from_i64<T>(a_ms), win);
  const T w = div_zero_rn(from_i64<T>(w_ms), win);
  T den = add_rn(a, mul_rn(wq, w));
  if (den < (T)1) den = (T)1;                       // demand floor of one request
  return div_zero_rn(num, den);
}

// sixteen bytes of values: four floats, or half of four doubles
template <class T> struct __align__(16) Four {
  T v[16 / sizeof(T)];
};

// STAGES: the two series of the stage-aware signal, each from its own counts
// (c0: prompt tokens over the prefill gauge and W with a token weight of one;
// c1: decode tokens over the decode gauge), read at the series' own elements;
// a null array counts as zeros.
template <class T, bool MEAN, int EPT, bool STAGES>
__global__ void __launch_bounds__(kEwThreads)
k_raw(const __grid_constant__ SeriesTable<T> tab, const __grid_constant__ TilePlan tp, FastDiv fm,
      bool vec, bool vec_w, Counts c0, Counts c1, const T* __restrict__ w_p, const T* __restrict__ w_q,
      T* __restrict__ raw, uint8_t* __restrict__ cls) {
  const int s = prefix_index(tp.tile_base, tab.n, blockIdx.x);
  const int M = tab.M;
  const int64_t n = (int64_t)tab.K[s] * M;
  const int64_t l0 = ((int64_t)(blockIdx.x - tp.tile_base[s]) * blockDim.x + threadIdx.x) * EPT;
  if (l0 >= n) return;
  const size_t x0 = (size_t)(tab.off[s] + l0);
  const Counts c = STAGES && s == 1 ? c1 : c0;
  const size_t xi = STAGES ? (size_t)l0 : x0;
  const T dt = div_rn((T)tab.win[s], (T)1000);      // window length in seconds
  int32_t p[EPT], d[EPT], a[EPT], w[EPT];
  long long am[EPT], wm[EPT];
  const bool v4 = EPT == 4 && vec && l0 + 4 <= n;
  if constexpr (EPT == 4) if (v4) {
    auto quad = [&](const int32_t* src, int32_t (&v)[EPT]) {
      const int4 q = !STAGES || src ? *reinterpret_cast<const int4*>(src + xi)
                                    : make_int4(0, 0, 0, 0);
      v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
    };
    quad(c.P, p);
    quad(c.D, d);
    if (MEAN) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const longlong2 A2 = reinterpret_cast<const longlong2*>(c.A_ms + xi)[h];
        const longlong2 W2 = reinterpret_cast<const longlong2*>(c.W_ms + xi)[h];
        am[2 * h] = A2.x; am[2 * h + 1] = A2.y;
        wm[2 * h] = W2.x; wm[2 * h + 1] = W2.y;
      }
    } else {
      quad(c.A, a);
      quad(c.W, w);
    }
  }
  if (!v4) {
#pragma unroll
    for (int i = 0; i < EPT; ++i) {
      const bool in = l0 + i < n;
      p[i] = in && (!STAGES || c.P) ? c.P[xi + i] : 0;
      d[i] = in && (!STAGES || c.D) ? c.D[xi + i] : 0;
      if (MEAN) {
        am[i] = in ? c.A_ms[xi + i] : 0;
        wm[i] = in ? c.W_ms[xi + i] : 0;
      } else {
        a[i] = in ? c.A[xi + i] : 0;
        w[i] = in && (!STAGES || c.W) ? c.W[xi + i] : 0;
      }
    }
  }
  int m = l0 <= 0xffffffffll ? (int)((uint32_t)l0 - fm.div((uint32_t)l0) * (uint32_t)M)
                             : (int)(l0 % M);
  // the weights of the elements' models: four in a row where M is a multiple of
  // four (m then is one too), else one by one
  T wp[EPT], wq[EPT];
  if (EPT == 4 && vec_w) {
#pragma unroll
    for (int h = 0; h < 4; h += 16 / (int)sizeof(T)) {
      const Four<T> a = *reinterpret_cast<const Four<T>*>(w_p + m + h);
      const Four<T> b = *reinterpret_cast<const Four<T>*>(w_q + m + h);
#pragma unroll
      for (int i = 0; i < 16 / (int)sizeof(T); ++i) {
        wp[(h + i) % EPT] = a.v[i];
        wq[(h + i) % EPT] = b.v[i];
      }
    }
  } else {
#pragma unroll
    for (int i = 0; i < EPT; ++i) {
      wp[i] = w_p[m];
      wq[i] = w_q[m];
      if (++m == M) m = 0;
    }
  }
  T rv[EPT];
  uint8_t cv[EPT];
#pragma unroll
  for (int i = 0; i < EPT; ++i) {
    bool idle;
    if (MEAN) {
      idle = (p[i] | d[i]) == 0 && (am[i] | wm[i]) == 0;
      rv[i] = idle ? idle_raw((T)0)
                   : raw_tss_mean<T>(p[i], d[i], am[i], wm[i], dt, (T)tab.win[s], wp[i], wq[i]);
    } else {
      idle = (p[i] | d[i] | a[i] | w[i]) == 0;
      rv[i] = idle ? idle_raw((T)0)
                   : raw_tss<T>(p[i], d[i], a[i], w[i], dt, STAGES && s == 0 ? (T)1 : wp[i],
                                wq[i]);
    }
    cv[i] = idle ? kIdle : kNom;
  }
  if constexpr (EPT == 4) {
    if (v4) {
#pragma unroll
      for (int h = 0; h < 4; h += 16 / (int)sizeof(T)) {
        Four<T> o;
#pragma unroll
        for (int i = 0; i < 16 / (int)sizeof(T); ++i) o.v[i] = rv[h + i];
        *reinterpret_cast<Four<T>*>(raw + x0 + h) = o;
      }
      *reinterpret_cast<uchar4*>(cls + x0) = make_uchar4(cv[0], cv[1], cv[2], cv[3]);
    }
  }
  if (!v4) {
#pragma unroll
    for (int i = 0; i < EPT; ++i)
      if (l0 + i < n) {
        raw[x0 + i] = rv[i];
        cls[x0 + i] = cv[i];
      }
  }
}

// raw values and classes of windows [k, k + kBatch) clipped to k1 (idle past k1)
template <class T>
__device__ __forceinline__ void load_batch(const T* __restrict__ raw, const uint8_t* __restrict__ cls,
                                           size_t base, int M, int64_t k, int64_t k1,
                                           T (&r)[kBatch], uint8_t (&c)[kBatch]) {
  if (k + kBatch <= k1) {
#pragma unroll
    for (int j = 0; j < kBatch; ++j) {
      const size_t x = base + (size_t)(k + j) * M;
      c[j] = cls[x];
      r[j] = raw[x];
    }
  } else {
#pragma unroll
    for (int j = 0; j < kBatch; ++j) {
      c[j] = kIdle;
      r[j] = (T)0;
      if (k + j < k1) {
        const size_t x = base + (size_t)(k + j) * M;
        c[j] = cls[x];
        r[j] = raw[x];
      }
    }
  }
}

// Run windows [k0, k1) of model m exactly from (S, init), writing S. With
// `verify`, stop at the first window whose new S equals the stored one with the
// same init state: from there the stored trajectory is the one this start
// produces. Returns true if it stopped early.
template <class T>
__device__ __forceinline__ bool run_segment(size_t base, int M, int64_t k0, int64_t k1,
                                            const T* __restrict__ raw, const ModelParams<T>& q,
                                            T& S, int& init, bool verify, int stored_init,
                                            T* S_out, const uint8_t* __restrict__ cls) {
  T r[kBatch], rn[kBatch];
  uint8_t c[kBatch], cn[kBatch];
  load_batch(raw, cls, base, M, k0, k1, r, c);
  for (int64_t k = k0; k < k1; k += kBatch) {
    T old[kBatch];
    if (verify) {
#pragma unroll
      for (int j = 0; j < kBatch; ++j)
        if (k + j < k1) old[j] = S_out[base + (size_t)(k + j) * M];
    }
    // next batch in flight while this one runs
    load_batch(raw, cls, base, M, k + kBatch, k1, rn, cn);
#pragma unroll
    for (int j = 0; j < kBatch; ++j) {
      if (k + j >= k1) break;
      if (c[j] != kIdle) {
        if (!init) {
          S = r[j];
          init = 1;
        } else {
          S = add_rn(mul_rn(q.a, r[j]), mul_rn(q.b, S));
        }
        stored_init = 1;
      }
      if (verify && init == stored_init && same_bits(S, old[j])) return true;
      S_out[base + (size_t)(k + j) * M] = init ? S : (T)0;
    }
#pragma unroll
    for (int j = 0; j < kBatch; ++j) {
      r[j] = rn[j];
      c[j] = cn[j];
    }
  }
  return false;
}

// ---- non-idle windows per (chunk, model) ----------------------------------
// One CTA per chunk: its windows are consecutive rows of [K][M], read 16 bytes
// at a time; idle windows are counted per model in shared memory.
template <class T>
__global__ void __launch_bounds__(256)
k_active(const __grid_constant__ SeriesTable<T> tab, FastDiv fm, const uint8_t* __restrict__ cls,
         int32_t* __restrict__ active) {
  extern __shared__ int32_t s_idle[];
  const int seg = blockIdx.x;
  const int s = series_of_seg(tab, seg);
  const int M = tab.M, L = tab.seg_len[s];
  const int64_t k0 = (int64_t)(seg - tab.seg_base[s]) * L, k1 = min64(k0 + L, tab.K[s]);
  for (int m = threadIdx.x; m < M; m += blockDim.x) s_idle[m] = 0;
  __syncthreads();
  const uint8_t* base = cls + tab.off[s] + (size_t)k0 * M;
  const uint32_t n = (uint32_t)((k1 - k0) * M);
  // bytes before the first 16-byte boundary, then whole 16-byte words, then the rest
  const uint32_t head = min(n, (uint32_t)((16 - ((uintptr_t)base & 15)) & 15));
  const uint32_t n16 = (n - head) / 16;
  auto count = [&](uint32_t i, uint8_t v) {
    if (v == kIdle) atomicAdd(&s_idle[i - fm.div(i) * (uint32_t)M], 1);
  };
  for (uint32_t i = threadIdx.x; i < head; i += blockDim.x) count(i, base[i]);
  const uint4* q = reinterpret_cast<const uint4*>(base + head);
  for (uint32_t w = threadIdx.x; w < n16; w += blockDim.x) {
    const uint4 v = q[w];
    const uint32_t ws[4] = {v.x, v.y, v.z, v.w};
    // a word with no idle byte needs no per-byte work
    bool any = false;
#pragma unroll
    for (int h = 0; h < 4; ++h) any |= __vcmpeq4(ws[h], kIdle * 0x01010101u) != 0;
    if (!any) continue;
    const uint32_t i0 = head + 16 * w;
#pragma unroll
    for (int h = 0; h < 4; ++h)
#pragma unroll
      for (int j = 0; j < 4; ++j) count(i0 + 4 * h + j, (uint8_t)(ws[h] >> (8 * j)));
  }
  for (uint32_t i = head + 16 * n16 + threadIdx.x; i < n; i += blockDim.x) count(i, base[i]);
  __syncthreads();
  const int rows = (int)(n / (uint32_t)M);
  for (int m = threadIdx.x; m < M; m += blockDim.x)
    active[(size_t)seg * M + m] = rows - s_idle[m];
}

// ---- pass 1: burn-in and chunk run, one lane per (chunk, model) -------------
// A CTA runs 32 chains, one per lane, in groups of kGroup windows. Three warps
// load the groups in turn and lay them in shared memory, one stage each; one runs
// the recurrences and writes S to shared memory; one stores S. They meet at named
// barriers, a pair per stage, so that none waits for another's whole group. The
// dependent chain is what bounds it (a product and a sum a window: 8.6 cycles in
// float, 128 in double, whose products and sums take 64 cycles each on this part
// and do not overlap within a warp), so its warp does little else: it moves four
// (in double two) windows with one 16-byte shared-memory access (a 4-byte store a
// window cost as much as the chain), and in double the product with alpha is the
// loaders' (warps 1 to 3 sit on other schedulers, with FP64 units of their own).
// One warp that copied, ran and stored took 37 cycles a window in float, 270 in
// double: 3 models, 600 windows in double 69 us, now 30.5; 8 models, 36,000
// windows in float 10.5, now 8.1; 64 models, 864,000 windows 204, now 149.
constexpr int kChains = 32;        // chains per CTA
constexpr int kLoaders = 3;
constexpr int kEmaThreads = 32 * (kLoaders + 2);
constexpr int kGroup = 32;         // windows per group
constexpr int kMaxBurn = 16384;    // burn-in cap (tiny alpha: the in-order pass repairs)
constexpr int64_t kActiveMinCells = 1 << 22;   // series cells from which burn-ins skip idle chunks
constexpr int64_t kEmaChains = 32768;         // (chunk, model) chains a long table is cut into
constexpr int64_t kShortChains = 16384;       // most chains a table is cut into by short chunks
// chunk and burn-in lengths are multiples of the group; short chunks are one
// group in double, two in float, where a chain's start costs as much as a group
template <class T> constexpr int short_chunk() { return sizeof(T) == 8 ? kGroup : 2 * kGroup; }

// Burn-in length, in updates (non-idle windows): (1 - alpha)^B <= e^-c, in
// whole groups, with c well past the point where a start error falls
// below the type's last bit, so that the rounded trajectories have met
// (c = 28 for float's 6e-8 = e^-16.6, 45 for double's 1.1e-16 = e^-36.7)
template <class T> __device__ __forceinline__ int burn_in(T alpha) {
  const float a = (float)alpha;
  const float c = sizeof(T) == 4 ? 28.f : 45.f;
  int B = kMaxBurn;
  if (a >= 1.f) B = kGroup;
  else if (a > 0.f) {
    const float x = c / -log1pf(-a);
    if (x < (float)kMaxBurn) B = (int)x + 1;
  }
  return (B + kGroup - 1) / kGroup * kGroup;
}

// The chain's input for one window: raw, or in double alpha * raw
template <class T> constexpr bool kPremul = sizeof(T) == 8;

// Consecutive windows of one chain, moved together; a stage holds [kGroup / V]
// rows of one such quad (pair) per chain.
template <class T> struct __align__(16) Windows {
  static constexpr int V = 16 / sizeof(T);
  T x[V];
};

// One group of windows of the chains; idle windows (and the padding of a lane's
// missing groups) carry the marker and leave S as it is. x: the chain's input,
// raw: the Eq. 1 values. STARTED: every lane has seen a non-idle window; STORE:
// write S.
template <class T, bool STARTED, bool STORE>
__device__ __forceinline__ void ema_group(const Windows<T>* x, const Windows<T>* raw,
                                          Windows<T>* dst, const ModelParams<T>& q, T& S,
                                          int& init) {
  constexpr int V = Windows<T>::V, N = kGroup / V;
  Windows<T> v[N];
#pragma unroll
  for (int h = 0; h < N; ++h) v[h] = x[h * kChains];
#pragma unroll
  for (int h = 0; h < N; ++h) {
    Windows<T> o;
#pragma unroll
    for (int j = 0; j < V; ++j) {
      const T in = v[h].x[j];
      const bool idle = is_idle_raw(in);
      const T nxt = add_rn(kPremul<T> ? in : mul_rn(q.a, in), mul_rn(q.b, S));
      if (STARTED) {
        S = idle ? S : nxt;
      } else if (!idle) {
        S = init ? nxt : raw[h * kChains].x[j];
        init = 1;
      }
      o.x[j] = S;                              // 0 until the chain starts
    }
    if (STORE) dst[h * kChains] = o;
  }
}

// Named barriers between one warp that fills (or empties) a stage and one that
// waits for it.
__device__ __forceinline__ void pair_wait(int id) {
  asm volatile("bar.sync %0, 64;\n" ::"r"(id) : "memory");
}
__device__ __forceinline__ void pair_arrive(int id) {
  asm volatile("bar.arrive %0, 64;\n" ::"r"(id) : "memory");
}
constexpr int kFullBar = 1, kEmptyBar = kFullBar + kLoaders;      // input stages
constexpr int kOutFullBar = kEmptyBar + kLoaders, kOutEmptyBar = kOutFullBar + 2;
static_assert(kOutEmptyBar + 2 <= 16, "named barriers of a CTA");

// stages of a buffer: the chain's inputs and, in double, the raw values too
template <class T> constexpr int ema_smem_bytes() {
  return (kLoaders * (kPremul<T> ? 2 : 1) + 2) * kGroup * kChains * (int)sizeof(T);
}

template <class T>
__global__ void __launch_bounds__(kEmaThreads)
k_ema(const __grid_constant__ SeriesTable<T> tab, const T* __restrict__ raw, const T* alpha,
      const T* S_carry, const uint8_t* init_carry, const int32_t* __restrict__ active,
      T* __restrict__ b_S, int32_t* __restrict__ b_init, T* __restrict__ e_S,
      int32_t* __restrict__ e_init, T* __restrict__ S_out) {
  extern __shared__ __align__(16) unsigned char ema_smem[];
  constexpr int V = Windows<T>::V, kStage = kGroup / V * kChains;
  Windows<T>* inb = reinterpret_cast<Windows<T>*>(ema_smem);    // [kLoaders] stages of inputs
  Windows<T>* rawb = kPremul<T> ? inb + kLoaders * kStage : inb;   // raw values
  Windows<T>* outb = rawb + kLoaders * kStage;                  // [2] stages of S
  const int M = tab.M;
  const int lane = threadIdx.x & 31, role = threadIdx.x >> 5;
  const int64_t t = (int64_t)blockIdx.x * kChains + lane;
  const bool has = t < (int64_t)tab.seg_base[tab.n] * M;  // a last CTA's spare lanes stay idle
  const int m = has ? (int)(t % M) : 0;
  const int seg = has ? (int)(t / M) : 0;
  const int s = series_of_seg(tab, seg);
  const ModelParams<T> q = load_params(tab, s, m, alpha);
  const int L = tab.seg_len[s];
  const int64_t k0 = (int64_t)(seg - tab.seg_base[s]) * L, k1 = min64(k0 + L, tab.K[s]);
  const int B = burn_in(q.a);
  // The burn-in runs over spans of windows [sp_lo, sp_hi), ascending. Without
  // activity counts it is the one span [k0 - B, k0). With them (non-idle
  // windows per chunk) it walks back over the preceding chunks until they hold
  // B non-idle windows, leaving out chunks that are wholly idle: an idle window
  // leaves the state as it is, so the trajectory is the same without them,
  // and a burn-in across a long idle stretch still sees enough updates.
  constexpr int kSpans = 8;
  int64_t sp_lo[kSpans], sp_hi[kSpans];
  int nsp = 0;
  bool from_start = false;   // the burn-in covers every update since window 0
  if (active == nullptr) {
    int64_t kb = k0 - B;
    if (kb <= 0) {
      kb = 0;
      from_start = true;
    }
    if (kb < k0) {
      sp_lo[0] = kb;
      sp_hi[0] = k0;
      nsp = 1;
    }
  } else {
    int64_t acc = 0;
    int cb = seg - tab.seg_base[s];
    const int32_t* act = active + (size_t)tab.seg_base[s] * M + m;
    while (acc < B) {
      if (cb == 0) {
        from_start = true;
        break;
      }
      --cb;
      const int na = act[(size_t)cb * M];
      if (na == 0) continue;
      const int64_t hi = (int64_t)(cb + 1) * L;   // chunks before this one are whole
      int64_t lo = (int64_t)cb * L;
      if (na == L && acc + L > B)
        lo = hi - (B - acc + kGroup - 1) / kGroup * kGroup;
      acc += na == L ? hi - lo : na;
      if (nsp > 0 && sp_lo[nsp - 1] == hi) {
        sp_lo[nsp - 1] = lo;
      } else if (nsp < kSpans) {
        sp_lo[nsp] = lo;
        sp_hi[nsp] = hi;
        ++nsp;
      } else {
        break;   // out of spans: a shorter burn-in, repaired by the in-order pass if short
      }
    }
    for (int i = 0; i < nsp / 2; ++i) {
      const int64_t l = sp_lo[i], h = sp_hi[i];
      sp_lo[i] = sp_lo[nsp - 1 - i];
      sp_hi[i] = sp_hi[nsp - 1 - i];
      sp_lo[nsp - 1 - i] = l;
      sp_hi[nsp - 1 - i] = h;
    }
  }
  const size_t base = (size_t)tab.off[s] + m;
  int burn = 0;                                     // groups of the burn-in
  for (int i = 0; i < nsp; ++i) burn += (int)((sp_hi[i] - sp_lo[i]) / kGroup);
  int own = (int)((k1 - k0 + kGroup - 1) / kGroup);  // groups of the chunk
  if (!has) burn = own = nsp = 0;
  // the lanes' chunks start together: a lane with a shorter burn-in waits
  const int lead = (int)__reduce_max_sync(0xffffffffu, (unsigned)burn);
  const int n_it = lead + (int)__reduce_max_sync(0xffffffffu, (unsigned)own);

  if (role == 0) {
    // the recurrences
    T S = (T)0;
    int init = has ? 0 : 1;                         // spare lanes do not hold the others up
    if (has && from_start) {                        // begin from the true state
      init = (init_carry && init_carry[m]) ? 1 : 0;
      S = init ? S_carry[m] : (T)0;
    }
    int stage = 0;
    for (int i = 0; i < n_it; ++i) {
      if (i == lead && has) {
        b_S[t] = S;
        b_init[t] = init;
      }
      const bool started = __all_sync(0xffffffffu, init);
      const int at = stage * kStage + lane;
      pair_wait(kFullBar + stage);
      if (i < lead) {
        if (started) ema_group<T, true, false>(inb + at, rawb + at, nullptr, q, S, init);
        else ema_group<T, false, false>(inb + at, rawb + at, nullptr, q, S, init);
      } else {
        const int o = (i - lead) & 1;
        Windows<T>* dst = outb + o * kStage + lane;
        if (i - lead >= 2) pair_wait(kOutEmptyBar + o);
        if (started) ema_group<T, true, true>(inb + at, rawb + at, dst, q, S, init);
        else ema_group<T, false, true>(inb + at, rawb + at, dst, q, S, init);
        pair_arrive(kOutFullBar + o);
      }
      if (i + kLoaders < n_it) pair_arrive(kEmptyBar + stage);
      stage = stage + 1 == kLoaders ? 0 : stage + 1;
    }
    if (has) {
      e_S[t] = S;
      e_init[t] = init;
    }
  } else if (role <= kLoaders) {
    // loader w fills stage w with groups w, w + 3, ...; the next kAhead of them
    // are on their way in registers
    constexpr int kAhead = sizeof(T) == 4 ? 2 : 1;
    T buf[kAhead][kGroup];
    auto load = [&](int gi, T (&v)[kGroup]) {
      int64_t k = k0, left = 0;
      int li = gi - (lead - burn);
      if (gi >= lead) {
        k = k0 + (int64_t)(gi - lead) * kGroup;
        left = gi < lead + own ? k1 - k : 0;
      } else if (li >= 0) {
        for (int i = 0; i < nsp; ++i) {             // span lengths are multiples of kGroup
          const int ng = (int)((sp_hi[i] - sp_lo[i]) / kGroup);
          if (li < ng) {
            k = sp_lo[i] + (int64_t)li * kGroup;
            left = kGroup;
            break;
          }
          li -= ng;
        }
      }
      const T* src = raw + base + (size_t)k * M;
      if (left >= kGroup) {
#pragma unroll
        for (int j = 0; j < kGroup; ++j) v[j] = __ldg(src + (size_t)j * M);
      } else {
#pragma unroll
        for (int j = 0; j < kGroup; ++j) v[j] = j < left ? __ldg(src + (size_t)j * M) : idle_raw((T)0);
      }
    };
    const int w = role - 1, at = w * kStage + lane;
#pragma unroll
    for (int h = 0; h < kAhead; ++h)
      if (w + h * kLoaders < n_it) load(w + h * kLoaders, buf[h]);
    for (int g0 = w; g0 < n_it; g0 += kAhead * kLoaders) {
#pragma unroll
      for (int h = 0; h < kAhead; ++h) {
        const int gi = g0 + h * kLoaders;
        if (gi < n_it) {
          if (gi >= kLoaders) pair_wait(kEmptyBar + w);
#pragma unroll
          for (int j = 0; j < kGroup; j += V) {
            Windows<T> r, x;
#pragma unroll
            for (int u = 0; u < V; ++u) {
              r.x[u] = buf[h][j + u];
              x.x[u] = is_idle_raw(r.x[u]) ? r.x[u] : mul_rn(q.a, r.x[u]);
            }
            rawb[at + j / V * kChains] = r;
            if (kPremul<T>) inb[at + j / V * kChains] = x;
          }
          pair_arrive(kFullBar + w);
          if (gi + kAhead * kLoaders < n_it) load(gi + kAhead * kLoaders, buf[h]);
        }
      }
    }
  } else {
    // stores
    T* out = S_out + base + (size_t)k0 * M;
    for (int gi = 0; gi < n_it - lead; ++gi) {
      const int o = gi & 1;
      pair_wait(kOutFullBar + o);
      const Windows<T>* src = outb + o * kStage + lane;
      const int64_t n = gi < own ? k1 - k0 - (int64_t)gi * kGroup : 0;
      T* d = out + (size_t)gi * kGroup * M;
#pragma unroll
      for (int j = 0; j < kGroup; j += V) {
        const Windows<T> v = src[j / V * kChains];
#pragma unroll
        for (int u = 0; u < V; ++u)
          if (j + u < n) d[(size_t)(j + u) * M] = v.x[u];
      }
      if (gi + 2 < n_it - lead) pair_arrive(kOutEmptyBar + o);
    }
  }
}

// ---- pass 2: boundary check and repair, one CTA per (series, model) ---------
// The CTA compares every chunk's burn-in state with its predecessor's end state
// (one round of loads; a warp that took 32 boundaries at a time waited on
// memory once per 32). Where none differs, as almost always, that is all. Else it
// repairs in passes: each chunk whose start differs is run again from its
// predecessor's end, a chunk a thread, until its new trajectory meets the stored
// one. A pass carries the states one chunk further, and a start error shrinks with
// every non-idle window on the way, so where burn-ins fell short because windows
// were idle here and there some passes make all starts equal the ends before them,
// which is the sequential result. From the share of idle windows that the first
// pass sees, the CTA reckons how many that takes; where they would cost more than
// half of a walk in order (long idle stretches, a tiny alpha), one lane walks. 8
// models, 36,000 windows, every other one idle, alpha 0.2: 128 us a call in float,
// 651 in double; 1,813 and 8,254 with one dry run before the walk in order,
// in which chunks had to meet within their own 64 or 32 windows.
constexpr int kResolveThreads = 128;
constexpr int kRerun = 2;          // start_init: the chunk has been run again
template <class T>
__global__ void __launch_bounds__(kResolveThreads)
k_resolve(const __grid_constant__ SeriesTable<T> tab, const T* __restrict__ raw, const T* alpha,
          T* start_S, int32_t* start_init, T* end_S, int32_t* end_init, T* S_out,
          const uint8_t* __restrict__ cls, T* S_carry, uint8_t* init_carry, tre_diag* diag) {
  __shared__ int first_s, seen_s[2];
  const int M = tab.M;
  const int s = blockIdx.x / M, m = blockIdx.x % M;
  const int n_seg = tab.seg_base[s + 1] - tab.seg_base[s];
  if (n_seg == 0) return;
  const size_t g0 = (size_t)tab.seg_base[s] * M + m;
  const int L = tab.seg_len[s];
  const size_t base = (size_t)tab.off[s] + m;
  // chunk c's state before it (its predecessor's end) and at its own start
  struct Edge {
    T pS;
    int pI, sI;
    bool bad;
  };
  auto edge = [&](int c) {
    const size_t x = g0 + (size_t)c * M;
    Edge e;
    e.pS = end_S[x - M];
    e.pI = end_init[x - M];
    e.sI = start_init[x];
    e.bad = (e.sI & 1) != e.pI || !same_bits(start_S[x], e.pS);
    return e;
  };
  bool differs = false;
#pragma unroll 4
  for (int c = 1 + threadIdx.x; c < n_seg; c += kResolveThreads) differs |= edge(c).bad;
  if (!__syncthreads_or(differs)) {
    if (S_carry && threadIdx.x == 0) {
      const size_t last = g0 + (size_t)(n_seg - 1) * M;
      S_carry[m] = end_S[last];
      init_carry[m] = (uint8_t)end_init[last];
    }
    return;
  }
  const ModelParams<T> q = load_params(tab, s, m, alpha);
  unsigned n_rerun = 0;
  bool some = true;
  const int rounds = (n_seg - 2) / kResolveThreads + 1;   // of a pass
  if (threadIdx.x < 2) seen_s[threadIdx.x] = 0;
  for (int pass = 0, n_pass = 1; pass < n_pass && some; ++pass) {
    some = false;
    int windows = 0, on = 0;       // of the chunks that met nothing stored
    for (int c0 = 1; c0 < n_seg; c0 += kResolveThreads) {
      const int c = c0 + (int)threadIdx.x;
      Edge e = {};
      if (c < n_seg) e = edge(c);
      // every thread has its predecessor's end before any of them changes
      if (!__syncthreads_or(e.bad)) continue;
      some = true;
      if (e.bad) {
        const size_t x = g0 + (size_t)c * M;
        const int64_t k0 = (int64_t)c * L, k1 = min64(k0 + L, tab.K[s]);
        T S = e.pS;
        int init = e.pI;
        const bool met =
            run_segment<T>(base, M, k0, k1, raw, q, S, init, true, e.sI & 1, S_out, cls);
        start_S[x] = e.pS;
        start_init[x] = e.pI | kRerun;
        if (!met) {
          end_S[x] = S;
          end_init[x] = init;
          if (pass == 0) {
            windows += (int)(k1 - k0);
#pragma unroll 8
            for (int64_t k = k0; k < k1; ++k) on += cls[base + (size_t)k * M] != kIdle;
          }
        }
        n_rerun += !(e.sI & kRerun);
      }
      __syncthreads();
    }
    if (pass == 0 && some) {
      if (windows) atomicAdd(&seen_s[0], windows);
      if (on) atomicAdd(&seen_s[1], on);
      __syncthreads();
      // updates that the burn-ins lacked, over those of a chunk; and two passes for
      // chunks with fewer than the mean
      const float w = (float)seen_s[0], u = (float)seen_s[1];
      const float passes = 2.f + (float)burn_in(q.a) * (w - u) / (u * (float)L);
      if (!(u < w)) n_pass = 2;
      else if (passes * (float)(2 * rounds) <= (float)n_seg) n_pass = 2 + (int)passes;
    }
  }
  if (n_rerun) atomicAdd(&diag->ema_resolved, (unsigned long long)n_rerun);
  int first_bad = n_seg;   // the in-order walk starts here
  if (some) {
    if (threadIdx.x == 0) first_s = n_seg;
    __syncthreads();
    for (int c = 1 + (int)threadIdx.x; c < n_seg; c += kResolveThreads)
      if (edge(c).bad) {
        atomicMin(&first_s, c);
        break;
      }
    __syncthreads();
    first_bad = first_s;
  }
  if (threadIdx.x != 0) return;
  const size_t last = g0 + (size_t)(first_bad - 1) * M;
  T S = end_S[last];
  int init = end_init[last];
  n_rerun = 0;
  for (int q0 = first_bad; q0 < n_seg; q0 += kBatch) {
    // load the boundary states of a batch of segments ahead of the checks
    T bS[kBatch], bE[kBatch];
    int bI[kBatch], bEI[kBatch];
#pragma unroll
    for (int j = 0; j < kBatch; ++j) {
      if (q0 + j < n_seg) {
        const size_t x = g0 + (size_t)(q0 + j) * M;
        bS[j] = start_S[x];
        bI[j] = start_init[x];
        bE[j] = end_S[x];
        bEI[j] = end_init[x];
      }
    }
#pragma unroll
    for (int j = 0; j < kBatch; ++j) {
      const int qq = q0 + j;
      if (qq >= n_seg) break;
      if (init == (bI[j] & 1) && same_bits(S, bS[j])) {
        S = bE[j];
        init = bEI[j];
        continue;
      }
      const int64_t k0 = (int64_t)qq * L, k1 = min64(k0 + L, tab.K[s]);
      const bool met =
          run_segment<T>(base, M, k0, k1, raw, q, S, init, true, bI[j] & 1, S_out, cls);
      if (met) {
        S = bE[j];
        init = bEI[j];
      }
      n_rerun += !(bI[j] & kRerun);
    }
  }
  if (n_rerun) atomicAdd(&diag->ema_resolved, (unsigned long long)n_rerun);
  if (S_carry) {
    S_carry[m] = S;
    init_carry[m] = (uint8_t)init;
  }
}

// ---- Z and regions from S ----------------------------------------------------
template <class T>
__device__ __forceinline__ uint8_t region_of(uint8_t idle, T z, T tc, T ts) {
  if (idle == kIdle) return kIdle;
  return z < tc ? kCrit : (z > ts ? kSurp : kNom);
}

// for every series of a table, elements in tiles as above
template <class T, int EPT>
__global__ void __launch_bounds__(kEwThreads)
k_normalize(const __grid_constant__ SeriesTable<T> tab, const __grid_constant__ TilePlan tp,
            FastDiv fm, bool vec, const T* S, const uint8_t* idle_cls, const T* theta,
            const T* tau_crit, T tau_crit_v, const T* tau_surp, T* Z, uint8_t* cls) {
  const int s = prefix_index(tp.tile_base, tab.n, blockIdx.x);
  const int M = tab.M;
  const int64_t n = (int64_t)tab.K[s] * M;
  const int64_t l0 =
      ((int64_t)(blockIdx.x - tp.tile_base[s]) * blockDim.x + threadIdx.x) * EPT;
  if (l0 >= n) return;
  const size_t x0 = (size_t)(tab.off[s] + l0);
  const bool v4 = EPT == 4 && vec && l0 + 4 <= n;
  T sv[EPT];
  uint8_t ic[EPT];
#pragma unroll
  for (int i = 0; i < EPT; ++i) sv[i] = v4 || l0 + i < n ? S[x0 + i] : (T)0;
  if constexpr (EPT == 4)
    if (v4) {
      const uchar4 c4 = *reinterpret_cast<const uchar4*>(idle_cls + x0);
      ic[0] = c4.x; ic[1] = c4.y; ic[2] = c4.z; ic[3] = c4.w;
    }
  if (!v4) {
#pragma unroll
    for (int i = 0; i < EPT; ++i) ic[i] = l0 + i < n ? idle_cls[x0 + i] : kIdle;
  }
  int m = l0 <= 0xffffffffll ? (int)((uint32_t)l0 - fm.div((uint32_t)l0) * (uint32_t)M)
                             : (int)(l0 % M);
  T zv[EPT];
  uint8_t cv[EPT];
#pragma unroll
  for (int i = 0; i < EPT; ++i) {
    zv[i] = div_rn(sv[i], theta[(size_t)s * M + m]);
    cv[i] = region_of(ic[i], zv[i], tau_crit ? tau_crit[m] : tau_crit_v, tau_surp[m]);
    if (++m == M) m = 0;
  }
#pragma unroll
  for (int i = 0; i < EPT; ++i) {
    if (!v4 && l0 + i >= n) break;
    if (Z) Z[x0 + i] = zv[i];
    if (cls && !v4) cls[x0 + i] = cv[i];
  }
  if constexpr (EPT == 4)
    if (cls && v4) *reinterpret_cast<uchar4*>(cls + x0) = make_uchar4(cv[0], cv[1], cv[2], cv[3]);
}

template <class T> __device__ __forceinline__ void load_quad_z(const T* p, T (&v)[4]);
template <> __device__ __forceinline__ void load_quad_z<float>(const float* p, float (&v)[4]) {
  const float4 q = *reinterpret_cast<const float4*>(p);
  v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
}
template <> __device__ __forceinline__ void load_quad_z<double>(const double* p, double (&v)[4]) {
  const double2 a = reinterpret_cast<const double2*>(p)[0];
  const double2 c = reinterpret_cast<const double2*>(p)[1];
  v[0] = a.x; v[1] = a.y; v[2] = c.x; v[3] = c.y;
}

// Z as an unsigned key in the order of the values (-0 as 0); any NaN comes after
// every value, and all ones, for an idle model, after that. Comparisons of
// doubles would take the pipe that their divisions wait for.
__device__ __forceinline__ uint32_t z_key(float z) {
  const uint32_t u = __float_as_uint(z);
  if ((u << 1) > 0xff000000u) return ~0u - 1u;
  return u == 0x80000000u ? u : u ^ ((u >> 31) ? ~0u : 0x80000000u);
}
__device__ __forceinline__ unsigned long long z_key(double z) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(z);
  if ((u << 1) > 0xffe0000000000000ull) return ~0ull - 1ull;
  return u == 0x8000000000000000ull ? u : u ^ ((u >> 63) ? ~0ull : 0x8000000000000000ull);
}
template <class T> struct ZKey;
template <> struct ZKey<float> { using U = uint32_t; };
template <> struct ZKey<double> { using U = unsigned long long; };
__device__ __forceinline__ uint32_t lowest_key(uint32_t k) {
  return __reduce_min_sync(0xffffffffu, k);
}
__device__ __forceinline__ unsigned long long lowest_key(unsigned long long k) {
  const uint32_t hi = (uint32_t)(k >> 32), h = __reduce_min_sync(0xffffffffu, hi);
  const uint32_t l = __reduce_min_sync(0xffffffffu, hi == h ? (uint32_t)k : ~0u);
  return (unsigned long long)h << 32 | l;
}

// One series with the Eq. 3 receiver per window: argmin Z over non-idle models,
// lowest index on ties (the first minimum in index order; a NaN only where it is
// the first model that is not idle), -1 when every model is idle. A CTA takes wt
// whole windows, their Z in shared memory (padded rows). Up to kRowThread models
// one thread per window scans its row, above that a warp: 48 models, 130,000
// windows in float 24.3 us by threads, 29.7 by warps; 72 models 30.6 and 28.3; 96
// models 29.4 and 25.1; 1,000 models, 10,000 windows 140 and 40 (double 327 and 189;
// 1,137 when the threads compared doubles). Bound in double by the divisions.
constexpr int kNormCells = 1024;
constexpr int kRowThread = 64;
constexpr int kNormQuadPasses = 4;
constexpr int kNoQuad = 0x7fffffff;
template <class T>
__global__ void __launch_bounds__(kEwThreads)
k_norm_recv(int M, int K, int wt, FastDiv fm, bool vec, const T* S,
            const uint8_t* idle_cls, const T* __restrict__ theta, const T* __restrict__ tau_crit,
            const T* __restrict__ tau_surp, T* Z, uint8_t* cls, int32_t* __restrict__ recv) {
  using U = typename ZKey<T>::U;
  constexpr U kIdleKey = ~(U)0, kNanKey = ~(U)0 - 1;
  // values of a float row that one thread scans, else keys: a comparison of floats
  // costs no more, and making keys does
  const bool values = sizeof(T) == 4 && M <= kRowThread;
  __shared__ U zs[2 * kNormCells];                     // [wt][M + 1]
  __shared__ uint8_t on[sizeof(T) == 4 ? 2 * kNormCells : 1];   // values: not idle
  const int k0 = (int)min64((int64_t)blockIdx.x * wt, K);
  const int nw = min(wt, K - k0), n = nw * M;
  const size_t x0 = (size_t)k0 * M;
  auto one = [&](int c, T sv, uint8_t ic, T& z, uint8_t& cl) {
    const int w = (int)fm.div((uint32_t)c), m = c - w * M;
    z = div_rn(sv, theta[m]);
    cl = region_of(ic, z, tau_crit[m], tau_surp[m]);
    const int at = w * (M + 1) + m;
    if constexpr (sizeof(T) == 4)
      if (values) {
        zs[at] = __float_as_uint(z);
        on[at] = cl != kIdle;
        return;
      }
    zs[at] = cl != kIdle ? z_key(z) : kIdleKey;
  };
  if (vec) {                                           // wt * M is a multiple of 4
    for (int c = 4 * threadIdx.x; c < n; c += 4 * blockDim.x) {
      T sv[4], z[4];
      load_quad_z<T>(S + x0 + c, sv);
      const uchar4 c4 = *reinterpret_cast<const uchar4*>(idle_cls + x0 + c);
      uint8_t cl[4];
      one(c, sv[0], c4.x, z[0], cl[0]);
      one(c + 1, sv[1], c4.y, z[1], cl[1]);
      one(c + 2, sv[2], c4.z, z[2], cl[2]);
      one(c + 3, sv[3], c4.w, z[3], cl[3]);
#pragma unroll
      for (int i = 0; i < 4; ++i) Z[x0 + c + i] = z[i];
      *reinterpret_cast<uchar4*>(cls + x0 + c) = make_uchar4(cl[0], cl[1], cl[2], cl[3]);
    }
  } else {
    for (int c = threadIdx.x; c < n; c += blockDim.x) {
      T z;
      uint8_t cl;
      one(c, S[x0 + c], idle_cls[x0 + c], z, cl);
      Z[x0 + c] = z;
      cls[x0 + c] = cl;
    }
  }
  __syncthreads();
  if (M <= kRowThread) {
    for (int w = threadIdx.x; w < nw; w += blockDim.x) {
      int best = -1;
      if constexpr (sizeof(T) == 4) {
        float low = 0.f;
#pragma unroll 8
        for (int m = 0; m < M; ++m) {
          const float z = __uint_as_float(zs[w * (M + 1) + m]);
          if (on[w * (M + 1) + m] && (best < 0 || z < low)) {
            best = m;
            low = z;
          }
        }
      } else {
        U low = kIdleKey;
#pragma unroll 8
        for (int m = 0; m < M; ++m) {
          const U k = zs[w * (M + 1) + m];
          if (k < low) {
            best = m;
            low = k == kNanKey ? (U)0 : k;             // nothing is lower than a first NaN
          }
        }
      }
      recv[k0 + w] = best;
    }
    return;
  }
  const int lane = threadIdx.x & 31;
  for (int w = threadIdx.x >> 5; w < nw; w += blockDim.x >> 5) {
    int best = kNoQuad, first = kNoQuad;               // first: low bit for a NaN
    U low = kIdleKey;
#pragma unroll 4
    for (int m = lane; m < M; m += 32) {
      const U k = zs[w * (M + 1) + m];
      if (k != kIdleKey && first == kNoQuad) first = 2 * m + (k == kNanKey ? 1 : 0);
      if (k < low) {
        best = m;
        low = k;
      }
    }
    const U l = lowest_key(low);
    best = __reduce_min_sync(0xffffffffu, low == l ? best : kNoQuad);
    first = __reduce_min_sync(0xffffffffu, first);
    if (lane == 0) recv[k0 + w] = first == kNoQuad ? -1 : first & 1 ? first >> 1 : best;
  }
}

// The same on large tables whose rows are 1, 2, 4, ... 32 quads of models: a
// thread keeps its quad of models (their theta and thresholds in registers) and
// takes one window after another, four in flight; a window's receiver comes from
// shuffles among the lanes that hold its row. A scan of the row by one thread left
// 240 of a CTA's 256 threads idle (64 models, 864,000 windows: 173 us, now 138). Bound by
// memory and by the division's instructions. Float only: in double k_norm_recv is
// faster (6.4 M cells: 122 us for 148, whatever the row's length).
__global__ void __launch_bounds__(kEwThreads)
k_norm_quads(int lg_quads, int64_t n_quads, const float* S, const uint8_t* idle_cls,
             const float* __restrict__ theta, const float* __restrict__ tau_crit,
             const float* __restrict__ tau_surp, float* Z, uint8_t* cls,
             int32_t* __restrict__ recv) {
  constexpr int U = kNormQuadPasses;
  const unsigned full = 0xffffffffu;
  const int64_t q0 = (int64_t)blockIdx.x * (kEwThreads * U) + threadIdx.x;
  const int lanes = 1 << lg_quads, m0 = 4 * (threadIdx.x & (lanes - 1));
  float th[4], tc[4], ts[4], sv[U][4];
  uchar4 ic[U];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    th[i] = theta[m0 + i];
    tc[i] = tau_crit[m0 + i];
    ts[i] = tau_surp[m0 + i];
  }
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const int64_t q = q0 + u * kEwThreads;
    ic[u] = make_uchar4(kIdle, kIdle, kIdle, kIdle);
#pragma unroll
    for (int i = 0; i < 4; ++i) sv[u][i] = 1.f;
    if (q < n_quads) {
      load_quad_z<float>(S + 4 * q, sv[u]);
      ic[u] = *reinterpret_cast<const uchar4*>(idle_cls + 4 * q);
    }
  }
#pragma unroll
  for (int u = 0; u < U; ++u) {
    const int64_t q = q0 + u * kEwThreads;
    const uint8_t idle[4] = {ic[u].x, ic[u].y, ic[u].z, ic[u].w};
    uint8_t cl[4];
    // the lowest value that is no NaN and its first model; the first model that is
    // not idle, with a low bit for a NaN (an ascending scan starts from it and
    // nothing compares below a NaN)
    int best = kNoQuad, first = kNoQuad;
    float bz = 0.f;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float z = div_zero_rn(sv[u][i], th[i]);
      sv[u][i] = z;
      cl[i] = region_of(idle[i], z, tc[i], ts[i]);
      const bool on = cl[i] != kIdle, nan = z != z;
      if (on && first == kNoQuad) first = 2 * (m0 + i) + (nan ? 1 : 0);
      if (on && !nan && (best == kNoQuad || z < bz)) {
        best = m0 + i;
        bz = z;
      }
    }
    if (q < n_quads) {
      *reinterpret_cast<float4*>(Z + 4 * q) = make_float4(sv[u][0], sv[u][1], sv[u][2], sv[u][3]);
      *reinterpret_cast<uchar4*>(cls + 4 * q) = make_uchar4(cl[0], cl[1], cl[2], cl[3]);
    }
    for (int o = 1; o < lanes; o <<= 1) {
      const int ob = __shfl_xor_sync(full, best, o);
      const float oz = __shfl_xor_sync(full, bz, o);
      if (ob != kNoQuad && (best == kNoQuad || oz < bz || (oz == bz && ob < best))) {
        best = ob;
        bz = oz;
      }
    }
    if (__any_sync(full, first != kNoQuad && (first & 1))) {
      for (int o = 1; o < lanes; o <<= 1) first = min(first, __shfl_xor_sync(full, first, o));
      if (first != kNoQuad && (first & 1)) best = first >> 1;
    }
    if (q < n_quads && m0 == 0) recv[q >> lg_quads] = best == kNoQuad ? -1 : best;
  }
}

// ---- per-window donor preference order (Sec. IV-B), warp per window ---------
// Donor key: group (idle 0, surplus 1, nominal above the receiver 2), then Z
// descending within surplus and nominal, then index. Keys are distinct, so the
// r-th donor is the smallest key above the (r-1)-th: kRankDonors rounds of a
// warp-wide minimum, each over the models whose key exceeds the last one.
template <class T>
__device__ __forceinline__ bool donor_key_less(int ga, T za, int ia, int gb, T zb, int ib) {
  if (ga != gb) return ga < gb;
  if (ga != 0 && za != zb) return za > zb;
  return ia < ib;
}

template <class T>
__global__ void k_rank(int M, int K, const T* Z, const uint8_t* cls, int32_t* recv,
                       int32_t* donors) {
  const int64_t k = (int64_t)blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32;
  if (k >= K) return;
  const int lane = threadIdx.x & 31;
  const T* z = Z + (size_t)k * M;
  const uint8_t* c = cls + (size_t)k * M;
  int best = -1;
  T bz = (T)0;
  for (int m = lane; m < M; m += 32) {
    if (c[m] == kIdle) continue;
    const T zm = z[m];
    if (best < 0 || zm < bz) { best = m; bz = zm; }
  }
  for (int o = 16; o > 0; o >>= 1) {
    const int ob = __shfl_xor_sync(0xffffffffu, best, o);
    const T oz = __shfl_xor_sync(0xffffffffu, bz, o);
    if (ob >= 0 && (best < 0 || oz < bz || (oz == bz && ob < best))) { best = ob; bz = oz; }
  }
  if (lane == 0 && recv) recv[k] = best;
  if (!donors) return;
  int32_t* out = donors + (size_t)k * kRankDonors;
  int lg = -1, li = -1;
  T lzv = (T)0;
  int r = 0;
  for (; best >= 0 && r < kRankDonors; ++r) {
    int g = 3, i = -1;
    T zv = (T)0;
    for (int m = lane; m < M; m += 32) {
      if (m == best) continue;
      const uint8_t cm = c[m];
      const T zm = z[m];
      int gm;
      if (cm == kIdle) gm = 0;
      else if (cm == kSurp) gm = 1;
      else if (cm == kNom && zm > bz) gm = 2;
      else continue;
      if (lg >= 0 && !donor_key_less(lg, lzv, li, gm, zm, m)) continue;
      if (i < 0 || donor_key_less(gm, zm, m, g, zv, i)) { g = gm; zv = zm; i = m; }
    }
    for (int o = 16; o > 0; o >>= 1) {
      const int og = __shfl_xor_sync(0xffffffffu, g, o);
      const int oi = __shfl_xor_sync(0xffffffffu, i, o);
      const T oz = __shfl_xor_sync(0xffffffffu, zv, o);
      if (oi >= 0 && (i < 0 || donor_key_less(og, oz, oi, g, zv, i))) { g = og; zv = oz; i = oi; }
    }
    if (i < 0) break;
    if (lane == 0) out[r] = i;
    lg = g; lzv = zv; li = i;
  }
  if (lane >= r && lane < kRankDonors) out[lane] = -1;
}

// Values of a rank: floats as they are; doubles, whose comparisons take the slow
// pipe, as unsigned keys in the same order (-0 as 0). Not for NaN.
template <class T> struct RankKey;
template <> struct RankKey<float> {
  float v;
  RankKey() = default;
  __device__ __forceinline__ explicit RankKey(float z) : v(z) {}
  __device__ __forceinline__ bool nan() const { return v != v; }
  static __device__ __forceinline__ RankKey most() { return RankKey(__int_as_float(0x7f800000)); }
};
template <> struct RankKey<double> {
  unsigned long long v;
  RankKey() = default;
  __device__ __forceinline__ explicit RankKey(double z) {
    const unsigned long long u = (unsigned long long)__double_as_longlong(z);
    v = u == 0x8000000000000000ull ? u : u ^ ((u >> 63) ? ~0ull : 0x8000000000000000ull);
  }
  __device__ __forceinline__ bool nan() const {    // outside the keys of both infinities
    return v - 0x000fffffffffffffull > 0xffe0000000000001ull;
  }
  static __device__ __forceinline__ RankKey most() {
    RankKey k;
    k.v = ~0ull;
    return k;
  }
};

// x << n, 0 from n = 32 on
__device__ __forceinline__ uint32_t shift_left(uint32_t x, uint32_t n) {
  uint32_t r;
  asm("shl.b32 %0, %1, %2;" : "=r"(r) : "r"(x), "r"(n));
  return r;
}

// One window by comparisons of its values, as an ascending scan orders them: for
// rows with a NaN among the models that are not idle.
template <class T>
__device__ __noinline__ void rank_window(int M, const T* z, const uint8_t* c, int32_t* recv,
                                         int32_t* out) {
  int best = -1;
  for (int m = 0; m < M; ++m)
    if (c[m] != kIdle && (best < 0 || z[m] < z[best])) best = m;
  if (recv) *recv = best;
  if (!out) return;
  for (int j = 0; j < kRankDonors; ++j) out[j] = -1;
  auto group = [&](int m) {
    if (m == best || best < 0) return 3;
    if (c[m] == kIdle) return 0;
    if (c[m] == kSurp) return 1;
    return c[m] == kNom && z[m] > z[best] ? 2 : 3;
  };
  for (int a = 0; a < M; ++a) {
    const int ga = group(a);
    if (ga == 3) continue;
    int r = 0;
    for (int b = 0; b < M; ++b) {
      const int gb = group(b);
      r += b != a && gb < 3 && donor_key_less(gb, z[b], b, ga, z[a], a);
    }
    if (r < kRankDonors) out[r] = a;
  }
}

// Up to 16 models: one thread per window, the row in registers. A donor's place is
// the number of donors of earlier groups and of those of its own group with a
// higher Z (the earlier index first on ties): every pair of values is compared
// once into a mask of the models before each, and groups are masks too. With QUAD
// (M a multiple of 4, 16-byte aligned arrays) rows are read four models a load; the
// eight donors leave in two 16-byte stores. Bound by instructions. 4 M windows of 8
// models in float: 147 us with 4-byte accesses 32 bytes apart and each pair
// compared twice on (group, Z, index), 98 with each compared once, now 72.
template <class T, int MMAX, bool QUAD>
__global__ void __launch_bounds__(256)
k_rank_small(int M, int K, const T* __restrict__ Z, const uint8_t* __restrict__ cls,
             int32_t* __restrict__ recv, int32_t* __restrict__ donors, bool store4) {
  static_assert(MMAX <= 16 && kRankDonors <= 8, "four bits a place, places in one word");
  static_assert(kCrit < 4 && kNom < 4 && kSurp < 4 && kIdle < 4, "two bits a region");
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= K) return;
  const T* z = Z + (size_t)k * M;
  const uint8_t* c = cls + (size_t)k * M;
  RankKey<T> zv[MMAX];
  uint32_t cv[MMAX];
#pragma unroll
  for (int m = 0; m < MMAX; m += 4) {
    if (QUAD && m < M) {
      T q[4];
      load_quad_z<T>(z + m, q);
      const uchar4 c4 = *reinterpret_cast<const uchar4*>(c + m);
#pragma unroll
      for (int i = 0; i < 4; ++i) zv[m + i] = RankKey<T>(q[i]);
      cv[m] = c4.x; cv[m + 1] = c4.y; cv[m + 2] = c4.z; cv[m + 3] = c4.w;
    } else {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const bool in = !QUAD && m + i < M;
        zv[m + i] = RankKey<T>(in ? z[m + i] : (T)0);
        cv[m + i] = in ? c[m + i] : kIdle;
      }
    }
  }
  // a mask per region, bit m for model m (a byte that is no region: none)
  uint32_t of[4] = {0, 0, 0, 0};
  const uint32_t all = (1u << M) - 1u;
  if (MMAX <= 8) {
    uint32_t w = 0;
#pragma unroll
    for (int m = 0; m < MMAX; ++m) w |= shift_left(1u << m, 8 * cv[m]);
#pragma unroll
    for (int r = 0; r < 4; ++r) of[r] = w >> (8 * r) & all;
  } else {
#pragma unroll
    for (int m = 0; m < MMAX; ++m)
#pragma unroll
      for (int r = 0; r < 4; ++r) of[r] |= cv[m] == (uint32_t)r ? 1u << m : 0u;
#pragma unroll
    for (int r = 0; r < 4; ++r) of[r] &= all;
  }
  const uint32_t idle = of[kIdle], busy = all & ~idle;
  // receiver: the lowest value of the models that are not idle
  bool odd = false;
  int best = -1;
  RankKey<T> bz = RankKey<T>::most();
#pragma unroll
  for (int m = 0; m < MMAX; ++m) {
    const bool on = busy >> m & 1u;
    odd |= on & zv[m].nan();
    if (on & (zv[m].v < bz.v)) {
      best = m;
      bz = zv[m];
    }
  }
  if (best < 0 && busy) best = __ffs(busy) - 1;      // nothing below infinity: the first
  int32_t* out = donors ? donors + (size_t)k * kRankDonors : nullptr;
  if (odd) {
    rank_window<T>(M, z, c, recv ? recv + k : nullptr, out);
    return;
  }
  if (recv) recv[k] = best;
  if (!donors) return;
  uint32_t before[MMAX], above = 0;
#pragma unroll
  for (int m = 0; m < MMAX; ++m) {
    before[m] = 0;
    if (bz.v < zv[m].v) above |= 1u << m;
  }
#pragma unroll
  for (int m = 1; m < MMAX; ++m)
#pragma unroll
    for (int q = 0; q < m; ++q) {
      if (zv[q].v >= zv[m].v) before[m] |= 1u << q;
      else before[q] |= 1u << m;
    }
  const uint32_t others = best >= 0 ? all & ~(1u << best) : 0u;
  const uint32_t g0 = idle & others, g1 = of[kSurp] & others, g2 = of[kNom] & others & above;
  const int n0 = __popc(g0), n1 = n0 + __popc(g1), n_don = n1 + __popc(g2);
  uint32_t low = 0;
#pragma unroll
  for (int m = 0; m < MMAX; ++m) {
    const uint32_t bit = 1u << m;
    const bool is0 = g0 & bit, is1 = g1 & bit, is2 = g2 & bit;
    const uint32_t ahead = is0 ? g0 & (bit - 1u) : before[m] & (is1 ? g1 : g2);
    const int at = __popc(ahead) + (is0 ? 0 : is1 ? n0 : n1);
    // four bits a place; no donor, or past the last place: shifted out
    low |= shift_left((uint32_t)m, is0 | is1 | is2 ? 4u * (uint32_t)at : 32u);
  }
  auto slot = [&](int j) -> int { return j < n_don ? (int)(low >> (4 * j) & 15u) : -1; };
  if (store4) {
#pragma unroll
    for (int j = 0; j < kRankDonors; j += 4)
      *reinterpret_cast<int4*>(out + j) = make_int4(slot(j), slot(j + 1), slot(j + 2), slot(j + 3));
  } else {
#pragma unroll
    for (int j = 0; j < kRankDonors; ++j) out[j] = slot(j);
  }
}

template <class T> TilePlan tile_plan(const SeriesTable<T>& t, int tile, int& n_tiles) {
  TilePlan tp;
  n_tiles = 0;
  for (int s = 0; s < t.n; ++s) {
    tp.tile_base[s] = n_tiles;
    n_tiles += (int)(((int64_t)t.K[s] * t.M + tile - 1) / tile);
  }
  tp.tile_base[t.n] = n_tiles;
  return tp;
}

// 16-byte accesses need every series to start on a 4-element boundary and
// the arrays on 16-byte ones
template <class T> bool quad_aligned(const SeriesTable<T>& t, std::initializer_list<const void*> ps) {
  for (int s = 0; s < t.n; ++s)
    if (t.off[s] % 4) return false;
  for (const void* p : ps)
    if (p && ((uintptr_t)p % 16)) return false;
  return true;
}

// four models' weights at a time: none of the fours wraps and all are aligned
inline bool weights_aligned(int M, const void* w_p, const void* w_q) {
  return M % 4 == 0 && (((uintptr_t)w_p | (uintptr_t)w_q) & 15) == 0;
}

template <class T> int64_t total_elems(const SeriesTable<T>& t) {
  int64_t n = 0;
  for (int s = 0; s < t.n; ++s) n += (int64_t)t.K[s] * t.M;
  return n;
}

}  // namespace

template <class T> int series_segments(SeriesTable<T>& t) {
  int total = 0;
  int64_t cells = 0;
  for (int s = 0; s < t.n; ++s) cells += (int64_t)t.K[s] * t.M;
  const bool few = cells / short_chunk<T>() <= kShortChains;
  for (int s = 0; s < t.n; ++s) {
    const int K = t.K[s];
    // A chain takes its burn-in plus its chunk, one window after another: short
    // chunks while the table gives few chains (three models, 600 windows in
    // double: 512 dependent steps with chunks of 256, 256 with 32), else 256
    // windows, longer for very long series (to bound the count) and for large
    // tables: about kEmaChains chains keep the GPU busy, and longer chunks
    // re-read fewer windows in their burn-ins. Multiples of the group.
    int L = few ? short_chunk<T>() : 256;
    int64_t need = std::max<int64_t>((K + 2047) / 2048, cells / kEmaChains);
    if (need > L) L = (int)((need + 2 * kGroup - 1) / (2 * kGroup) * (2 * kGroup));
    t.seg_len[s] = L;
    t.seg_base[s] = total;
    total += (K + L - 1) / L;
  }
  t.seg_base[t.n] = total;
  return total;
}

template <class T> void score_ws_layout(Arena& a, int M, int64_t elems, int n_seg, ScoreWs<T>& w) {
  w.raw = a.take<T>((size_t)std::max<int64_t>(elems, 1));
  w.cap_seg = std::max(n_seg, 1);
  const size_t n = (size_t)w.cap_seg * M;
  w.start_S = a.take<T>(n);
  w.start_init = a.take<int32_t>(n);
  w.end_S = a.take<T>(n);
  w.end_init = a.take<int32_t>(n);
  w.active = a.take<int32_t>(n);
}

template <class T> int score_launches(const SeriesTable<T>& tab, bool with_z) {
  return (total_elems(tab) >= kActiveMinCells ? 1 : 0) + 3 + (with_z ? 1 : 0);
}

// the smoothing of Eq. 1 values and idle classes k_raw has written
template <class T>
static cudaError_t smooth(const SeriesTable<T>& tab, const T* alpha, T* S_carry,
                          uint8_t* init_carry, T* S, const uint8_t* cls, ScoreWs<T>& w,
                          tre_diag* diag, cudaStream_t s) {
  const int M = tab.M;
  const int n_seg = tab.seg_base[tab.n];
  if (n_seg > w.cap_seg) return cudaErrorInvalidValue;
  const int64_t segs = (int64_t)n_seg * M;
  const unsigned g = (unsigned)((segs + kChains - 1) / kChains);
  // activity counts for the burn-ins where the series are long enough that
  // idle stretches would otherwise send chunks to the in-order pass, and the
  // extra pass over the classes is small beside the smoothing
  const int32_t* active = nullptr;
  if (total_elems(tab) >= kActiveMinCells) {
    k_active<T><<<n_seg, 256, (size_t)M * sizeof(int32_t), s>>>(tab, FastDiv(M), cls, w.active);
    active = w.active;
  }
  cudaError_t e = func_smem_once((const void*)k_ema<T>, ema_smem_bytes<T>(), false);
  if (e) return e;
  k_ema<T><<<g, kEmaThreads, ema_smem_bytes<T>(), s>>>(tab, w.raw, alpha, S_carry, init_carry,
                                                       active, w.start_S, w.start_init, w.end_S,
                                                       w.end_init, S);
  k_resolve<T><<<tab.n * M, kResolveThreads, 0, s>>>(tab, w.raw, alpha, w.start_S, w.start_init,
                                                     w.end_S, w.end_init, S, cls, S_carry,
                                                     init_carry, diag);
  return cudaGetLastError();
}

template <class T>
cudaError_t launch_score(const SeriesTable<T>& tab, const int32_t* P, const int32_t* D,
                         const int32_t* A, const int32_t* W, const T* w_p, const T* w_q,
                         const T* alpha, const T* theta, const T* tau_crit, const T* tau_surp,
                         T* S_carry, uint8_t* init_carry, T* S, T* Z, uint8_t* cls,
                         int32_t* recv, ScoreWs<T>& w, tre_diag* diag, cudaStream_t s,
                         const int64_t* A_ms, const int64_t* W_ms) {
  const int M = tab.M;
  if ((A_ms == nullptr) != (W_ms == nullptr)) return cudaErrorInvalidValue;
  const int64_t total = total_elems(tab);
  if (total == 0) return cudaSuccess;
  const Counts c{P, D, A, W, A_ms, W_ms};
  const bool small = total <= kSmallCells;
  const int th = small ? kSmallThreads : kEwThreads;
  int n_tiles = 0;
  const TilePlan tp = tile_plan(tab, small ? th : 4 * th, n_tiles);
  const bool vec_w = weights_aligned(M, w_p, w_q);
  if (A_ms) {
    const bool vec = quad_aligned(tab, {P, D, A_ms, W_ms, w.raw, cls});
    auto f = small ? k_raw<T, true, 1, false> : k_raw<T, true, 4, false>;
    f<<<n_tiles, th, 0, s>>>(tab, tp, FastDiv(M), vec, vec_w, c, c, w_p, w_q, w.raw, cls);
  } else {
    const bool vec = quad_aligned(tab, {P, D, A, W, w.raw, cls});
    auto f = small ? k_raw<T, false, 1, false> : k_raw<T, false, 4, false>;
    f<<<n_tiles, th, 0, s>>>(tab, tp, FastDiv(M), vec, vec_w, c, c, w_p, w_q, w.raw, cls);
  }
  const cudaError_t e = smooth<T>(tab, alpha, S_carry, init_carry, S, cls, w, diag, s);
  if (e) return e;
  // Z and regions in a pass of their own: the division in the chain's warp
  // cost more than re-reading S (8 models, 60 windows in double: 33 us of
  // smoothing with it; one hour of 100 ms windows in float: 42)
  if (theta) return launch_normalize<T>(tab, S, cls, theta, tau_crit, (T)0, tau_surp, Z, cls, recv, s);
  return cudaSuccess;
}

// The stage-aware signal as a table of two series (prefill, decode): Eq. 1 of
// each from its own counts, smoothed together; S, cls at the series' offsets.
template <class T>
cudaError_t launch_score_stages(const SeriesTable<T>& tab, const int32_t* P, const int32_t* D,
                                const int32_t* W, const int32_t* A_pre, const int32_t* A_dec,
                                const T* w_p, const T* w_q, const T* alpha, T* S, uint8_t* cls,
                                ScoreWs<T>& w, tre_diag* diag, cudaStream_t s) {
  const int64_t total = total_elems(tab);
  if (total == 0) return cudaSuccess;
  const bool small = total <= kSmallCells;
  const int th = small ? kSmallThreads : kEwThreads;
  int n_tiles = 0;
  const TilePlan tp = tile_plan(tab, small ? th : 4 * th, n_tiles);
  const Counts pre{P, nullptr, A_pre, W, nullptr, nullptr};
  const Counts dec{nullptr, D, A_dec, nullptr, nullptr, nullptr};
  const bool vec = quad_aligned(tab, {P, D, W, A_pre, A_dec, w.raw, cls});
  const bool vec_w = weights_aligned(tab.M, w_p, w_q);
  auto f = small ? k_raw<T, false, 1, true> : k_raw<T, false, 4, true>;
  f<<<n_tiles, th, 0, s>>>(tab, tp, FastDiv(tab.M), vec, vec_w, pre, dec, w_p, w_q, w.raw, cls);
  return smooth<T>(tab, alpha, nullptr, nullptr, S, cls, w, diag, s);
}

// both stages' S, Z and regions into arrays of their own (blockIdx.y: stage)
template <class T>
__global__ void __launch_bounds__(kSmallThreads)
k_norm_stages(const __grid_constant__ SeriesTable<T> tab, FastDiv fm, const T* __restrict__ S,
              const uint8_t* __restrict__ idle_cls, const T* __restrict__ tau_crit,
              const T* __restrict__ tau_surp, StageOut<T> o0, StageOut<T> o1) {
  const StageOut<T> o = blockIdx.y ? o1 : o0;
  const int M = tab.M;
  const int64_t n = (int64_t)tab.K[0] * M, off = tab.off[blockIdx.y];
  for (int64_t i = (int64_t)blockIdx.x * kSmallThreads + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * kSmallThreads) {
    const int m = i <= 0xffffffffll ? (int)((uint32_t)i - fm.div((uint32_t)i) * (uint32_t)M)
                                    : (int)(i % M);
    const T v = S[off + i], z = div_rn(v, o.theta[m]);
    o.S[i] = v;
    o.Z[i] = z;
    o.cls[i] = region_of(idle_cls[off + i], z, tau_crit[m], tau_surp[m]);
  }
}

template <class T>
cudaError_t launch_norm_stages(const SeriesTable<T>& tab, const T* S, const uint8_t* idle_cls,
                               const T* tau_crit, const T* tau_surp, const StageOut<T>& pre,
                               const StageOut<T>& dec, cudaStream_t s) {
  const int64_t n = (int64_t)tab.K[0] * tab.M;
  if (n == 0) return cudaSuccess;
  const int64_t b = std::min<int64_t>((n + kSmallThreads - 1) / kSmallThreads,
                                      (int64_t)device_sm_count() * 16);
  k_norm_stages<T><<<dim3((unsigned)b, 2), kSmallThreads, 0, s>>>(
      tab, FastDiv(tab.M), S, idle_cls, tau_crit, tau_surp, pre, dec);
  return cudaGetLastError();
}

template <class T>
cudaError_t launch_normalize(const SeriesTable<T>& tab, const T* S, const uint8_t* idle_cls,
                             const T* theta, const T* tau_crit, T tau_crit_v, const T* tau_surp,
                             T* Z, uint8_t* cls, int32_t* recv, cudaStream_t s) {
  const int64_t total = total_elems(tab);
  if (total == 0) return cudaSuccess;
  const bool small = total <= kSmallCells;
  const bool vec = quad_aligned(tab, {S, idle_cls, Z, cls});
  if (recv) {
    if (tab.n != 1 || !tau_crit || !Z || !cls) return cudaErrorInvalidValue;
    const int M = tab.M, K = tab.K[0], th = small ? kSmallThreads : kEwThreads;
    int lg_quads = 0;
    while (lg_quads < 5 && 4 << lg_quads < M) ++lg_quads;
    if constexpr (sizeof(T) == 4) {
      if (vec && !small && M == 4 << lg_quads) {
        constexpr int kPerCta = kEwThreads * kNormQuadPasses;
        const int64_t n_quads = (int64_t)K << lg_quads;
        k_norm_quads<<<(unsigned)((n_quads + kPerCta - 1) / kPerCta), kEwThreads, 0, s>>>(
            lg_quads, n_quads, S, idle_cls, theta, tau_crit, tau_surp, Z, cls, recv);
        return cudaGetLastError();
      }
    }
    const int wt = std::max(1, (small ? th : kNormCells) / M);
    k_norm_recv<T><<<(unsigned)((K + wt - 1) / wt), th, 0, s>>>(
        M, K, wt, FastDiv(M), vec && !small && M % 4 == 0, S, idle_cls, theta, tau_crit, tau_surp,
        Z, cls, recv);
    return cudaGetLastError();
  }
  int n_tiles = 0;
  const int th = small ? kSmallThreads : kEwThreads;
  const TilePlan tp = tile_plan(tab, small ? th : 4 * th, n_tiles);
  auto f = small ? k_normalize<T, 1> : k_normalize<T, 4>;
  f<<<n_tiles, th, 0, s>>>(tab, tp, FastDiv(tab.M), vec, S, idle_cls, theta, tau_crit, tau_crit_v,
                           tau_surp, Z, cls);
  return cudaGetLastError();
}

template <class T>
cudaError_t launch_rank(int M, int K, const T* Z, const uint8_t* cls, int32_t* recv,
                        int32_t* donors, cudaStream_t s) {
  if (K == 0 || (!recv && !donors)) return cudaSuccess;
  const unsigned thread_blocks = (unsigned)((K + 255) / 256);
  const bool quad = M % 4 == 0 && (((uintptr_t)Z | (uintptr_t)cls) & 15) == 0;
  const bool store4 = ((uintptr_t)donors & 15) == 0;
  if (M <= 16) {
    auto f = M <= 8 ? (quad ? k_rank_small<T, 8, true> : k_rank_small<T, 8, false>)
                    : (quad ? k_rank_small<T, 16, true> : k_rank_small<T, 16, false>);
    f<<<thread_blocks, 256, 0, s>>>(M, K, Z, cls, recv, donors, store4);
  }
  else
    k_rank<T><<<(unsigned)((K + 7) / 8), 256, 0, s>>>(M, K, Z, cls, recv, donors);
  return cudaGetLastError();
}

#define TRE_INST(T)                                                                               \
  template cudaError_t launch_score_stages<T>(const SeriesTable<T>&, const int32_t*,               \
                                              const int32_t*, const int32_t*, const int32_t*,      \
                                              const int32_t*, const T*, const T*, const T*, T*,    \
                                              uint8_t*, ScoreWs<T>&, tre_diag*, cudaStream_t);     \
  template cudaError_t launch_norm_stages<T>(const SeriesTable<T>&, const T*, const uint8_t*,      \
                                             const T*, const T*, const StageOut<T>&,               \
                                             const StageOut<T>&, cudaStream_t);                    \
  template int series_segments<T>(SeriesTable<T>&);                                               \
  template int score_launches<T>(const SeriesTable<T>&, bool);                                        \
  template void score_ws_layout<T>(Arena&, int, int64_t, int, ScoreWs<T>&);                       \
  template cudaError_t launch_score<T>(const SeriesTable<T>&, const int32_t*, const int32_t*,      \
                                       const int32_t*, const int32_t*, const T*, const T*,         \
                                       const T*, const T*, const T*, const T*, T*, uint8_t*, T*,   \
                                       T*, uint8_t*, int32_t*, ScoreWs<T>&, tre_diag*,             \
                                       cudaStream_t,                                               \
                                       const int64_t*, const int64_t*);                            \
  template cudaError_t launch_normalize<T>(const SeriesTable<T>&, const T*, const uint8_t*,        \
                                           const T*, const T*, T, const T*, T*, uint8_t*,          \
                                           int32_t*, cudaStream_t);                                \
  template cudaError_t launch_rank<T>(int, int, const T*, const uint8_t*, int32_t*, int32_t*,      \
                                      cudaStream_t);
TRE_INST(float)
TRE_INST(double)

}  // namespace tre
