// Open-loop TRE move selection (Sec. IV-B dual-speed control, Eq. 3 receiver,
// Sec. IV-C bounded pairwise transfer under a fixed budget).
//
// Everything that does not depend on the replica state is computed first, in
// parallel, for every (series, rescue threshold, control tick):
//   - at each fast tick: whether any model is critical, the rescue receiver
//     (lowest Z among critical models, lowest index on ties) and every model's
//     rank in the rescue donor order;
//   - at each slow tick: the Eq. 3 receiver over non-idle models, whether its
//     Z is below 1, and every model's rank in the rebalance donor order.
// Donor order: idle models by index, then surplus by Z descending, then
// nominal by Z descending (in rebalance only those above the receiver's Z);
// critical models and the receiver get no rank.
// The serial part walks the ticks with the replica counts in registers. On
// nested cadences (slow a multiple of fast, no fast tick shorter than a
// window) and up to 64 models it is k_walk_lane: a warp per controller
// instance, a model per lane, jumping from move to move. Other cadences visit
// every tick (k_walk_thread up to 16 models, k_walk above), as do more than 64
// models (k_walk).
#include <algorithm>
#include <cstddef>

#include "common.cuh"
#include "internal.h"

namespace tre {
namespace {

constexpr uint16_t kNoRank = 0xffff;

__device__ __forceinline__ int64_t tick_window(int64_t j, int64_t cadence, int64_t win) {
  // window whose right edge passes the j-th multiple of the cadence (j >= 1)
  return (j * cadence + win - 1) / win - 1;
}

// successive multiples j*c of a cadence c as quotient and remainder of win
struct TickSeq {
  int32_t q, r, qc, rc, win;
  __device__ __forceinline__ TickSeq(int32_t c, int32_t w) : win(w) {
    qc = c / w;
    rc = c - qc * w;
    q = qc;
    r = rc;
  }
  // window whose right edge passes the current multiple (windows end before 2^31 ms)
  __device__ __forceinline__ int32_t window() const { return q + (r > 0) - 1; }
  __device__ __forceinline__ void next() {
    q += qc;
    r += rc;
    if (r >= win) { r -= win; q += 1; }
  }
};

template <class T>
__device__ __forceinline__ uint8_t region_of(uint8_t c, T z, T tc, T ts) {
  if (c == kIdle) return kIdle;
  if (z < tc) return kCrit;
  if (z > ts) return kSurp;
  return kNom;
}

// One thread per (series, tau, tick entry, model). Entries [0, nf) of a series
// are its fast ticks, [nf, nf + ns) its slow ticks.
template <class T>
__global__ void __launch_bounds__(256)
k_tick_rank(const __grid_constant__ WalkBatch<T> b, int16_t* recv_out, int16_t* ndon_out,
            uint16_t* rank, uint16_t* order, unsigned long long* dm64) {
  const int M = b.M;
  const int64_t gid = (int64_t)blockIdx.x * 256 + threadIdx.x;
  const int64_t total_ent = (int64_t)b.ent_base[b.n_series] * b.n_tau;
  if (gid >= total_ent * M) return;
  const int m = (int)(gid % M);
  const int64_t e = gid / M;                       // entry over (series, tau, tick)
  const int s = prefix_index(b.ent_base, b.n_series, e, b.n_tau);
  const int64_t local = e - (int64_t)b.ent_base[s] * b.n_tau;
  const int n_ent = b.ent_base[s + 1] - b.ent_base[s];
  const int ti = (int)(local / n_ent);
  const int j = (int)(local % n_ent);
  const int64_t win = b.series_win[s];
  const int64_t K = b.series_K[s];
  const int64_t nf = K * win / b.fast_ms;
  const bool fast = j < nf;
  const int64_t k =
      fast ? tick_window(j + 1, b.fast_ms, win) : tick_window(j - nf + 1, b.slow_ms, win);
  const T* Zk = b.Z + b.series_off[s] + (size_t)k * M;
  const uint8_t* Ck = b.cls + b.series_off[s] + (size_t)k * M;
  const bool tau_dev = b.tau_crit != nullptr;
  const T tau_v = b.tau_list[tau_dev ? 0 : ti];
  auto reg = [&](int q) {
    return region_of(Ck[q], Zk[q], tau_dev ? b.tau_crit[q] : tau_v, b.tau_surp[q]);
  };
  // receiver: rescue -> lowest Z among critical; rebalance -> lowest Z among non-idle
  int recv = -1;
  T zr = (T)0;
  for (int q = 0; q < M; ++q) {
    const uint8_t rg = reg(q);
    const bool cand = fast ? rg == kCrit : rg != kIdle;
    if (cand && (recv < 0 || Zk[q] < zr)) {
      recv = q;
      zr = Zk[q];
    }
  }
  const bool act = recv >= 0 && (fast || zr < (T)1);
  // donor group of model q, -1 = not a donor at this tick
  auto group = [&](int q, uint8_t rg) -> int {
    if (q == recv || rg == kCrit) return -1;
    if (rg == kIdle) return 0;
    if (rg == kSurp) return 1;
    if (!fast && !(Zk[q] > zr)) return -1;       // rebalance: nominal donors above the receiver
    return 2;
  };
  const int gm = act ? group(m, reg(m)) : -1;
  uint16_t r = kNoRank;
  if (gm >= 0) {
    const T zm = Zk[m];
    int before = 0;
    for (int q = 0; q < M; ++q) {
      if (q == m) continue;
      const int gq = group(q, reg(q));
      if (gq < 0) continue;
      bool prec;
      if (gq != gm) prec = gq < gm;
      else if (gq == 0) prec = q < m;
      else prec = Zk[q] > zm || (Zk[q] == zm && q < m);
      before += prec;
    }
    r = (uint16_t)before;
  }
  const size_t row = (size_t)b.ent_base[s] * b.n_tau + (size_t)ti * n_ent + j;
  rank[row * M + m] = r;
  if (r != kNoRank) order[row * M + r] = (uint16_t)m;
  if (m == 0) {
    int nd = 0;
    unsigned long long dm = 0;
    if (act)
      for (int q = 0; q < M; ++q)
        if (group(q, reg(q)) >= 0) {
          ++nd;
          if (q < 64) dm |= 1ull << q;
        }
    recv_out[row] = (int16_t)(act ? recv : -1);
    ndon_out[row] = (int16_t)nd;
    if (dm64) dm64[row] = dm;                      // models that are donors at the tick
  }
}

__device__ __forceinline__ void load_quad(const float* p, float* v) {
  const float4 q = *reinterpret_cast<const float4*>(p);
  v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
}
__device__ __forceinline__ void load_quad(const double* p, double* v) {
  const double2 a = reinterpret_cast<const double2*>(p)[0];
  const double2 c = reinterpret_cast<const double2*>(p)[1];
  v[0] = a.x; v[1] = a.y; v[2] = c.x; v[3] = c.y;
}

// The action of one control tick of (series s, tau ti) at window k, for
// M <= MMAX: regions from the window's Z and class rows; the receiver (rescue:
// lowest Z among critical models; rebalance: lowest Z among non-idle models,
// acting only below Z = 1; lowest index on ties; -1 when the tick does
// nothing); each model's rank in the donor order (kNoRank when not a donor),
// the donor order packed four bits a position (M <= 16), the donor mask and
// the donor count.
template <class T, int MMAX>
struct TickAction {
  int recv, nd;
  unsigned long long pk, dmw;
  uint32_t dm;
  uint16_t rk[MMAX];
};

template <class T, int MMAX>
__device__ __forceinline__ void tick_row(const WalkBatch<T>& b, int s, uint32_t k, T (&z)[MMAX],
                                         uint8_t (&cl)[MMAX]) {
  const int M = b.M;
  const T* Zk = b.Z + b.series_off[s] + (size_t)k * M;
  const uint8_t* Ck = b.cls + b.series_off[s] + (size_t)k * M;
#pragma unroll
  for (int q = 0; q < MMAX; ++q) {
    z[q] = (T)0;
    cl[q] = kIdle;
  }
#pragma unroll
  for (int q = 0; q < MMAX; ++q)
    if (q < M) {
      z[q] = Zk[q];
      cl[q] = Ck[q];
    }
}

template <class T, int MMAX>
__device__ __forceinline__ void tick_action(const WalkBatch<T>& b, int ti, bool fast,
                                            const T (&z)[MMAX], const uint8_t (&cl)[MMAX],
                                            TickAction<T, MMAX>& out) {
  const int M = b.M;
  const bool tau_dev = b.tau_crit != nullptr;
  const T tau_v = b.tau_list[tau_dev ? 0 : ti];
  uint8_t rg[MMAX];
  int recv = -1;
  T zr = (T)0;
#pragma unroll
  for (int q = 0; q < MMAX; ++q) {
    rg[q] = 0xff;
    if (q < M) {
      rg[q] = region_of(cl[q], z[q], tau_dev ? b.tau_crit[q] : tau_v, b.tau_surp[q]);
      const bool cand = fast ? rg[q] == kCrit : rg[q] != kIdle;
      if (cand && (recv < 0 || z[q] < zr)) {
        recv = q;
        zr = z[q];
      }
    }
  }
  const bool act = recv >= 0 && (fast || zr < (T)1);
  int grp[MMAX];
  int nd = 0;
#pragma unroll
  for (int q = 0; q < MMAX; ++q) {
    int g = -1;
    if (act && q < M && q != recv && rg[q] != kCrit) {
      if (rg[q] == kIdle) g = 0;
      else if (rg[q] == kSurp) g = 1;
      else if (fast || z[q] > zr) g = 2;       // rebalance: nominal donors above the receiver
    }
    grp[q] = g;
    nd += g >= 0;
  }
  unsigned long long pk = 0, dmw = 0;
  uint32_t dm = 0;
#pragma unroll
  for (int m = 0; m < MMAX; ++m) {
    uint16_t r = kNoRank;
    if (m < M && grp[m] >= 0) {
      int before = 0;
#pragma unroll
      for (int q = 0; q < MMAX; ++q) {
        if (q >= M || q == m || grp[q] < 0) continue;
        bool prec;
        if (grp[q] != grp[m]) prec = grp[q] < grp[m];
        else if (grp[q] == 0) prec = q < m;
        else prec = z[q] > z[m] || (z[q] == z[m] && q < m);
        before += prec;
      }
      r = (uint16_t)before;
      dmw |= 1ull << m;
      if (MMAX <= 16) {
        pk |= (unsigned long long)m << (4 * before);
        dm |= 1u << m;
      }
    }
    out.rk[m] = r;
  }
  out.recv = act ? recv : -1;
  out.nd = nd;
  out.pk = pk;
  out.dm = dm;
  out.dmw = dmw;
}

// One thread per (series, tau, tick entry) for M <= MMAX: the regions are
// computed once per model and the ranks in registers; the per-model rank and
// order tables are written only when the walk that follows reads them.
template <class T, int MMAX>
__global__ void __launch_bounds__(128)
k_tick_rank_small(const __grid_constant__ WalkBatch<T> b, int16_t* recv_out, int16_t* ndon_out,
                  uint16_t* rank, uint16_t* order, unsigned long long* packed, uint32_t* dmask,
                  bool need_rank, unsigned long long* dm64) {
  const int M = b.M;
  const int64_t e = (int64_t)blockIdx.x * 128 + threadIdx.x;
  if (e >= (int64_t)b.ent_base[b.n_series] * b.n_tau) return;
  const int s = prefix_index(b.ent_base, b.n_series, e, b.n_tau);
  const int local = (int)(e - (int64_t)b.ent_base[s] * b.n_tau);
  const int n_ent = b.ent_base[s + 1] - b.ent_base[s];
  const int ti = local / n_ent;
  const int j = local - ti * n_ent;
  // K * win < 2^31, so every tick time below fits 32 unsigned bits
  const uint32_t win = (uint32_t)b.series_win[s];
  const uint32_t nf = (uint32_t)b.series_K[s] * win / (uint32_t)b.fast_ms;
  const bool fast = (uint32_t)j < nf;
  const uint32_t tj = fast ? ((uint32_t)j + 1) * (uint32_t)b.fast_ms
                           : ((uint32_t)j - nf + 1) * (uint32_t)b.slow_ms;
  const uint32_t k = (tj + win - 1) / win - 1;   // window whose right edge passes tj
  T z[MMAX];
  uint8_t cl[MMAX];
  tick_row<T, MMAX>(b, s, k, z, cl);
  TickAction<T, MMAX> a;
  tick_action<T, MMAX>(b, ti, fast, z, cl, a);
  const size_t row = (size_t)b.ent_base[s] * b.n_tau + (size_t)ti * n_ent + j;
  if (need_rank) {
#pragma unroll
    for (int m = 0; m < MMAX; ++m) {
      if (m >= M) break;
      rank[row * M + m] = a.rk[m];
      if (a.rk[m] != kNoRank) order[row * M + a.rk[m]] = (uint16_t)m;
    }
    dm64[row] = a.dmw;                             // for the warp walk
  }
  recv_out[row] = (int16_t)a.recv;
  ndon_out[row] = (int16_t)a.nd;
  if (MMAX <= 16) {
    packed[row] = a.pk;
    dmask[row] = a.dm;
  }
}

template <int MPL>
__device__ __forceinline__ int lane_of_min_rank(const uint16_t (&rk)[MPL], const int (&r)[MPL],
                                                const int (&rmin)[MPL], int lane, int M,
                                                int& model) {
  uint32_t best = 0xffffffffu;
  int bj = 0;
#pragma unroll
  for (int j = 0; j < MPL; ++j) {
    const bool ok = lane + 32 * j < M && rk[j] != kNoRank && r[j] > rmin[j];
    if (ok && rk[j] < best) {
      best = rk[j];
      bj = j;
    }
  }
  const uint32_t wmin = __reduce_min_sync(0xffffffffu, best);
  if (wmin == 0xffffffffu) return -1;
  const unsigned who = __ballot_sync(0xffffffffu, best == wmin);
  const int src = __ffs(who) - 1;            // ranks are distinct within a tick
  model = src + 32 * __shfl_sync(0xffffffffu, bj, src);
  return src;
}

// One CTA per (series, tau) and group of up to kCapWarps pacing caps, one warp
// per cap: the warps share the tick tables of their (series, tau), staged in
// shared memory when they fit. (Eight warps a CTA leave each thread the
// registers the walk's state needs.)
constexpr int kCapWarps = 8;
template <class T, int MPL, bool STAGED>
__global__ void __launch_bounds__(kCapWarps * 32)
k_walk(const __grid_constant__ WalkBatch<T> b, const int16_t* recv_tab, const int16_t* ndon_tab,
       const uint16_t* rank, const uint16_t* order, const unsigned long long* dm64) {
  extern __shared__ __align__(16) unsigned char dyn[];
  const int grp = blockIdx.x;                       // (series, tau)
  const int ti = grp % b.n_tau;
  const int si = grp / b.n_tau;
  const int ci = blockIdx.y * kCapWarps + threadIdx.x / 32;   // pacing cap index
  const int lane = threadIdx.x & 31;
  const int M = b.M;
  const int K = b.series_K[si];
  const int64_t win = b.series_win[si];
  const int n_ent = b.ent_base[si + 1] - b.ent_base[si];
  const size_t row0 = (size_t)b.ent_base[si] * b.n_tau + (size_t)ti * n_ent;
  const int16_t* rv_tab = recv_tab + row0;
  const int16_t* nd_tab = ndon_tab + row0;
  const unsigned long long* dm_tab = dm64 + row0;
  const uint16_t* rk0 = rank + row0 * M;
  const uint16_t* od0 = order + row0 * M;
  if (STAGED) {
    const size_t a2 = ((size_t)n_ent * 2 + 15) & ~(size_t)15;
    const size_t am = ((size_t)n_ent * M * 2 + 15) & ~(size_t)15;
    int16_t* srv = reinterpret_cast<int16_t*>(dyn);
    int16_t* snd = reinterpret_cast<int16_t*>(dyn + a2);
    uint16_t* srk = reinterpret_cast<uint16_t*>(dyn + 2 * a2);
    uint16_t* sod = reinterpret_cast<uint16_t*>(dyn + 2 * a2 + am);
    for (int i = threadIdx.x; i < n_ent; i += blockDim.x) {
      srv[i] = rv_tab[i];
      snd[i] = nd_tab[i];
    }
    for (int64_t i = threadIdx.x; i < (int64_t)n_ent * M; i += blockDim.x) {
      srk[i] = rk0[i];
      sod[i] = od0[i];
    }
    __syncthreads();
    rv_tab = srv;
    nd_tab = snd;
    rk0 = srk;
    od0 = sod;
  }
  if (ci >= b.n_cap) return;
  const int inst = (si * b.n_tau + ti) * b.n_cap + ci;
  const int Kp = b.cap_list[ci];
  const int64_t cap = b.moves_cap;
  tre_move* mv = b.moves + (size_t)inst * cap;
  const int64_t F = b.fast_ms, Sl = b.slow_ms;
  const int64_t nf = (int64_t)K * win / F;

  int r[MPL], rmin[MPL], g[MPL];
  int64_t used = 0;
  bool bad = false;
#pragma unroll
  for (int j = 0; j < MPL; ++j) {
    const int m = lane + 32 * j;
    if (m < M) {
      r[j] = b.r0[m];
      rmin[j] = b.r_min[m];
      g[j] = b.footprint[m];
      used += (int64_t)g[j] * r[j];
      if (r[j] < 0 || g[j] < 1 || rmin[j] < 0) bad = true;
    } else {
      r[j] = 0; rmin[j] = 0; g[j] = 0;
    }
  }
  for (int o = 16; o > 0; o >>= 1) used += __shfl_xor_sync(0xffffffffu, used, o);
  int64_t free_pool = b.budget - used;
  // an inconsistent controller state (negative replicas or floors, footprint
  // below one, replicas beyond the budget) produces no moves
  if (__any_sync(0xffffffffu, bad) || free_pool < 0) {
#pragma unroll
    for (int j = 0; j < MPL; ++j)
      if (lane + 32 * j < M) b.r_out[(size_t)inst * M + lane + 32 * j] = r[j];
    if (lane == 0) {
      b.n_moves[inst] = 0;
      b.diag->err = TRE_EINVAL;
    }
    return;
  }
  int64_t nm = 0;
  // With unit footprints and one model per lane a tick is closed form: pool
  // draws first, then donors drain in rank order down to their floors.
  bool unit = true;
#pragma unroll
  for (int j = 0; j < MPL; ++j)
    if (lane + 32 * j < M && g[j] != 1) unit = false;
  const bool closed = MPL == 1 && __all_sync(0xffffffffu, unit);
  // tick windows without division: the j-th tick of a cadence c ends window
  // ceil(j*c / win) - 1; keep j*c as quotient and remainder of win
  TickSeq sf((int32_t)F, (int32_t)win), ss((int32_t)Sl, (int32_t)win);
  int32_t jf = 1, js = 1;
  // the receivers of the coming 32 fast and 32 slow ticks, one per lane: most
  // ticks move nothing, and a tick then costs a shuffle instead of a load
  int32_t fb0 = -64, sb0 = -64;                 // entries >= 0: the first access loads
  int fbuf = -1, sbuf = -1;
  auto rv_at = [&](int32_t e, int32_t& b0, int& buf) {
    if ((uint32_t)(e - b0) >= 32u) {
      b0 = e;
      buf = e + lane < n_ent ? rv_tab[e + lane] : -1;
    }
    return __shfl_sync(0xffffffffu, buf, e - b0);
  };
  // the donor sets of the same ticks (models with a rank), for up to 64
  // models: a tick whose receiver the pool cannot serve and whose donors all
  // sit at their floors moves nothing, and costs no row load
  int32_t fm0 = -64, sm0 = -64;
  unsigned long long fmb = 0, smb = 0;
  auto dm_at = [&](int32_t e, int32_t& b0, unsigned long long& buf) {
    if ((uint32_t)(e - b0) >= 32u) {
      b0 = e;
      buf = e + lane < n_ent ? dm_tab[e + lane] : 0ull;
    }
    return __shfl_sync(0xffffffffu, buf, e - b0);
  };
  // the transitions of one tick: window k, receiver recv, table entry ent
  auto act = [&](int32_t k, int recv, int kind, int32_t ent) {
    if (closed) {
      const int nd = nd_tab[ent];
      const int mo = lane < nd ? od0[(size_t)ent * M + lane] : -1;
      const int r_src = __shfl_sync(0xffffffffu, r[0] - rmin[0], mo < 0 ? 0 : mo);
      const int cap_p = mo < 0 ? 0 : (r_src > 0 ? r_src : 0);
      int incl = cap_p;
      for (int o = 1; o < 32; o <<= 1) {
        const int x = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += x;
      }
      const int excl = incl - cap_p;
      const int total_cap = __shfl_sync(0xffffffffu, incl, 31);
      const int n_pool = (int)(free_pool < Kp ? free_pool : Kp);
      const int t_d = min(Kp - n_pool, total_cap);
      const int give = max(0, min(t_d - excl, cap_p));
      // moves: pool draws take seq 0.., donors follow in rank order
      for (int q = lane; q < n_pool; q += 32)
        if (nm + q < cap)
          mv[nm + q] = tre_move{(int32_t)k, (int16_t)recv, (int16_t)-1, (uint8_t)kind,
                                (uint8_t)q, 0};
      for (int i = 0; i < give; ++i) {
        const int64_t q = n_pool + excl + i;
        if (nm + q < cap)
          mv[nm + q] = tre_move{(int32_t)k, (int16_t)recv, (int16_t)mo, (uint8_t)kind,
                                (uint8_t)q, 0};
      }
      // my model's position in the donor order, then what it gave
      const uint16_t my_rank = lane < M ? rk0[(size_t)ent * M + lane] : kNoRank;
      const int given = __shfl_sync(0xffffffffu, give, my_rank == kNoRank ? 0 : (my_rank & 31));
      if (my_rank != kNoRank) r[0] -= given;
      if (lane == recv) r[0] += n_pool + t_d;
      free_pool -= n_pool;
      nm += n_pool + t_d;
      return;
    }
    uint16_t rk[MPL];
#pragma unroll
    for (int j = 0; j < MPL; ++j)
      rk[j] = lane + 32 * j < M ? rk0[(size_t)ent * M + lane + 32 * j] : kNoRank;
    int g_own = 0;
#pragma unroll
    for (int j = 0; j < MPL; ++j)
      if (lane + 32 * j == recv) g_own = g[j];
    const int need = __shfl_sync(0xffffffffu, g_own, recv & 31);
    for (int seq = 0; seq < Kp; ++seq) {
      if (free_pool >= need) {
        free_pool -= need;
#pragma unroll
        for (int j = 0; j < MPL; ++j)
          if (lane + 32 * j == recv) r[j] += 1;
        if (lane == 0 && nm < cap)
          mv[nm] = tre_move{(int32_t)k, (int16_t)recv, (int16_t)-1, (uint8_t)kind, (uint8_t)seq, 0};
        ++nm;
        continue;
      }
      // release donor replicas one at a time until the receiver's footprint
      // fits; an uncoverable transition releases nothing and ends the tick
      int rr[MPL];
#pragma unroll
      for (int j = 0; j < MPL; ++j) rr[j] = r[j];
      int64_t f = free_pool;
      const int64_t nm0 = nm;
      bool ok = true;
      while (f < need) {
        int d = -1;
        const int src = lane_of_min_rank<MPL>(rk, rr, rmin, lane, M, d);
        if (src < 0) { ok = false; break; }
        int gd = 0;
#pragma unroll
        for (int j = 0; j < MPL; ++j)
          if (lane + 32 * j == d) { rr[j] -= 1; gd = g[j]; }
        gd = __shfl_sync(0xffffffffu, gd, src);
        f += gd;
        if (lane == 0 && nm < cap)
          mv[nm] = tre_move{(int32_t)k, (int16_t)recv, (int16_t)d, (uint8_t)kind, (uint8_t)seq, 0};
        ++nm;
      }
      if (!ok) {
        nm = nm0;
        break;
      }
#pragma unroll
      for (int j = 0; j < MPL; ++j) {
        r[j] = rr[j];
        if (lane + 32 * j == recv) r[j] += 1;
      }
      free_pool = f - need;
    }
  };
  while (true) {
    const int32_t kf = sf.window(), ks = ss.window();
    const int32_t k = kf < ks ? kf : ks;
    if (k >= K) break;
    const bool fast = kf == k, slow = ks == k;
    const int32_t ef = jf - 1, es = (int32_t)nf + js - 1;   // entries of this tick
    while (sf.window() <= k) { sf.next(); ++jf; }
    while (ss.window() <= k) { ss.next(); ++js; }
    int recv = -1, kind = 0;
    int32_t ent = -1;
    if (fast) {
      const int rv = rv_at(ef, fb0, fbuf);
      if (rv >= 0) { recv = rv; ent = ef; kind = TRE_RESCUE; }
    }
    if (!kind && slow) {
      const int rv = rv_at(es, sb0, sbuf);
      if (rv >= 0) { recv = rv; ent = es; kind = TRE_REBALANCE; }
    }
    if (!kind) continue;
    if (MPL <= 2) {
      const unsigned long long donors =
          ent < (int32_t)nf ? dm_at(ent, fm0, fmb) : dm_at(ent, sm0, smb);
      unsigned long long above = 0;
#pragma unroll
      for (int j = 0; j < MPL; ++j)
        above |= (unsigned long long)__ballot_sync(0xffffffffu, lane + 32 * j < M && r[j] > rmin[j])
                 << (32 * j);
      int g_rv = 0;
#pragma unroll
      for (int j = 0; j < MPL; ++j)
        if (lane + 32 * j == recv) g_rv = g[j];
      const int need_rv = __shfl_sync(0xffffffffu, g_rv, recv & 31);
      if (free_pool < need_rv && !(donors & above)) continue;
    }
    act(k, recv, kind, ent);
  }
#pragma unroll
  for (int j = 0; j < MPL; ++j) {
    const int m = lane + 32 * j;
    if (m < M) b.r_out[(size_t)inst * M + m] = r[j];
  }
  if (lane == 0) {
    b.n_moves[inst] = nm;
    if (nm > cap) b.diag->err = TRE_EOVERFLOW;
  }
}

// One thread per controller instance (M <= 16): the threads of a CTA are the
// pacing caps of one (series, tau) and share its staged tick tables. A
// transition draws on the idle pool if it covers the receiver's footprint,
// else releases donor replicas in the tick's donor order (lowest rank first,
// each down to its floor). The models still above their floors are a bit
// mask in a register, so a tick whose donors are all at their floors costs one
// AND; the donor order is a packed 4-bit list per tick.
template <class T, int MMAX>
__device__ __forceinline__ int sel(const int (&a)[MMAX], int m) {
  int v = 0;
#pragma unroll
  for (int q = 0; q < MMAX; ++q) v = q == m ? a[q] : v;
  return v;
}
template <class T, int MMAX>
__device__ __forceinline__ void add_at(int (&a)[MMAX], int m, int d) {
#pragma unroll
  for (int q = 0; q < MMAX; ++q) a[q] += q == m ? d : 0;
}

template <class T, int MMAX>
__global__ void __launch_bounds__(32)
k_walk_thread(const __grid_constant__ WalkBatch<T> b, const int16_t* recv_tab,
              const unsigned long long* packed, const uint32_t* dmask) {
  extern __shared__ __align__(16) unsigned char dyn[];
  const int grp = blockIdx.x;
  const int ti = grp % b.n_tau;
  const int si = grp / b.n_tau;
  const int M = b.M;
  const int K = b.series_K[si];
  const int32_t win = b.series_win[si];
  const int n_ent = b.ent_base[si + 1] - b.ent_base[si];
  const size_t row0 = (size_t)b.ent_base[si] * b.n_tau + (size_t)ti * n_ent;
  unsigned long long* spk = reinterpret_cast<unsigned long long*>(dyn);
  uint32_t* sdm = reinterpret_cast<uint32_t*>(spk + n_ent);
  int16_t* srv = reinterpret_cast<int16_t*>(sdm + n_ent);
  for (int i = threadIdx.x; i < n_ent; i += blockDim.x) {
    spk[i] = packed[row0 + i];
    sdm[i] = dmask[row0 + i];
    srv[i] = recv_tab[row0 + i];
  }
  __syncthreads();
  const int ci = threadIdx.x;
  if (ci >= b.n_cap) return;
  const int inst = (si * b.n_tau + ti) * b.n_cap + ci;
  const int Kp = b.cap_list[ci];
  const int64_t cap = b.moves_cap;
  tre_move* mv = b.moves + (size_t)inst * cap;
  const int32_t nf = (int32_t)((int64_t)K * win / b.fast_ms);
  int r[MMAX], rmin[MMAX], g[MMAX];
  int64_t used = 0;
  bool bad = false, unit = true;
  uint32_t avail = 0;                           // models above their floor
#pragma unroll
  for (int m = 0; m < MMAX; ++m) {
    r[m] = 0;
    rmin[m] = 0;
    g[m] = 1;
    if (m < M) {
      r[m] = b.r0[m];
      rmin[m] = b.r_min[m];
      g[m] = b.footprint[m];
      used += (int64_t)g[m] * r[m];
      if (r[m] < 0 || rmin[m] < 0 || g[m] < 1) bad = true;
      if (g[m] != 1) unit = false;
      if (r[m] > rmin[m]) avail |= 1u << m;
    }
  }
  int64_t free_pool = b.budget - used;
  if (bad || free_pool < 0) {
    for (int m = 0; m < M && m < MMAX; ++m) b.r_out[(size_t)inst * M + m] = sel<T, MMAX>(r, m);
    b.n_moves[inst] = 0;
    b.diag->err = TRE_EINVAL;
    return;
  }
  auto emit = [&](int64_t at, int32_t k, int recv, int donor, int kind, int sq) {
    if (at < cap) mv[at] = tre_move{k, (int16_t)recv, (int16_t)donor, (uint8_t)kind, (uint8_t)sq, 0};
  };
  int64_t nm = 0;
  TickSeq sf(b.fast_ms, win), ss(b.slow_ms, win);
  int32_t jf = 1, js = 1;
  while (true) {
    const int32_t kf = sf.window(), ks = ss.window();
    const int32_t k = kf < ks ? kf : ks;
    if (k >= K) break;
    const bool fast = kf == k, slow = ks == k;
    const int32_t ef = jf - 1, es = nf + js - 1;
    while (sf.window() <= k) { sf.next(); ++jf; }
    while (ss.window() <= k) { ss.next(); ++js; }
    int recv = -1, kind = 0;
    int32_t ent = -1;
    if (fast) {
      const int rv = srv[ef];
      if (rv >= 0) { recv = rv; ent = ef; kind = TRE_RESCUE; }
    }
    if (!kind && slow) {
      const int rv = srv[es];
      if (rv >= 0) { recv = rv; ent = es; kind = TRE_REBALANCE; }
    }
    if (!kind) continue;
    const uint32_t usable = avail & sdm[ent];
    const int need = unit ? 1 : sel<T, MMAX>(g, recv);
    if (free_pool < need && !usable) continue;        // nothing can move this tick
    unsigned long long pk = spk[ent];
    if (unit) {
      const int n_pool = (int)(free_pool < Kp ? free_pool : Kp);
      for (int q = 0; q < n_pool; ++q) emit(nm + q, k, recv, -1, kind, q);
      int sq = n_pool;
      uint32_t left = usable;
      while (sq < Kp && left) {
        int m = (int)(pk & 15);                      // next model in donor order
        pk >>= 4;
        if (!(left >> m & 1)) continue;
        left &= ~(1u << m);
        const int c = sel<T, MMAX>(r, m) - sel<T, MMAX>(rmin, m);
        const int take = min(c, Kp - sq);
        add_at<T, MMAX>(r, m, -take);
        if (take == c) avail &= ~(1u << m);
        for (int i = 0; i < take; ++i, ++sq) emit(nm + sq, k, recv, m, kind, sq);
      }
      add_at<T, MMAX>(r, recv, sq);
      if (sel<T, MMAX>(r, recv) > sel<T, MMAX>(rmin, recv)) avail |= 1u << recv;
      free_pool -= n_pool;
      nm += sq;
      continue;
    }
    for (int sq = 0; sq < Kp; ++sq) {
      if (free_pool >= need) {
        free_pool -= need;
        add_at<T, MMAX>(r, recv, 1);
        if (sel<T, MMAX>(r, recv) > sel<T, MMAX>(rmin, recv)) avail |= 1u << recv;
        emit(nm++, k, recv, -1, kind, sq);
        continue;
      }
      // plan the releases; an uncoverable transition releases nothing
      int64_t f = free_pool;
      const int64_t nm0 = nm;
      int taken[MMAX];
#pragma unroll
      for (int m = 0; m < MMAX; ++m) taken[m] = 0;
      unsigned long long order = pk;
      uint32_t left = avail & sdm[ent];
      while (f < need && left) {
        const int m = (int)(order & 15);
        order >>= 4;
        if (!(left >> m & 1)) continue;
        left &= ~(1u << m);
        int c = sel<T, MMAX>(r, m) - sel<T, MMAX>(rmin, m);
        const int gm = sel<T, MMAX>(g, m);
        while (f < need && c > 0) {
          add_at<T, MMAX>(taken, m, 1);
          --c;
          f += gm;
          emit(nm++, k, recv, m, kind, sq);
        }
      }
      if (f < need) {
        nm = nm0;
        break;
      }
#pragma unroll
      for (int m = 0; m < MMAX; ++m) {
        r[m] -= taken[m];
        if (m < M && !(r[m] > rmin[m])) avail &= ~(1u << m);
      }
      add_at<T, MMAX>(r, recv, 1);
      if (sel<T, MMAX>(r, recv) > sel<T, MMAX>(rmin, recv)) avail |= 1u << recv;
      free_pool = f - need;
    }
  }
  for (int m = 0; m < M && m < MMAX; ++m) b.r_out[(size_t)inst * M + m] = sel<T, MMAX>(r, m);
  b.n_moves[inst] = nm;
  if (nm > cap) b.diag->err = TRE_EOVERFLOW;
}

// One move record, written as three 32-bit words (window; receiver and donor;
// kind and position in the tick) when it fits the caller's list.
static_assert(sizeof(tre_move) == 12 && offsetof(tre_move, recv) == 4 &&
                  offsetof(tre_move, donor) == 6 && offsetof(tre_move, kind) == 8 &&
                  offsetof(tre_move, seq) == 9 && offsetof(tre_move, reserved) == 10,
              "tre_move layout");
__device__ __forceinline__ void put_move(tre_move* mv, int64_t at, int64_t cap, int32_t k,
                                         int recv, int donor, int kind, int sq) {
  if (at < cap) {
    uint32_t* p = reinterpret_cast<uint32_t*>(mv + at);
    p[0] = (uint32_t)k;
    p[1] = (uint32_t)(uint16_t)recv | ((uint32_t)(uint16_t)donor << 16);
    p[2] = (uint32_t)(uint8_t)kind | ((uint32_t)(uint8_t)sq << 8);
  }
}

// ---- lane walk: nested cadences, up to 64 models ----------------------------
// On nested cadences the ticks are the fast ticks, and what a tick would do
// (receiver, kind, donor order) does not depend on the replica state, so the
// state only decides which tick moves something next: the first one where the
// idle pool is not empty or a donor stands above its floor. Ticks are cut into
// chunks of kChunk; k_tick_rows ranks a chunk's ticks and stores, per tick u of
// the chunk and model, one word (16 bits up to 16 models, else 32)
//     first tick t >= u of the chunk where the model is a donor | rank | receiver
// (rank from 1 in that tick's donor order; t = kChunk: none left in the chunk).
// k_walk_lane keeps one model per lane (two above 32): one shared-memory load
// of the row at u, masked by "above its floor", and one warp-wide minimum give
// the next tick that moves something and its donor together. Ranking and walk
// measured, before (one thread per tick; one lane jumping over tables of next
// donor ticks up to 16 models, one warp testing 32 ticks a ballot above) and
// now: 16 models, 4,320 ticks, 431 moves 228 -> 57 us; 64 models, 17,280
// ticks, 1,493 moves 1,504 -> 202 us; 24 models of unequal footprint, 720
// ticks, 1,875 moves 634 -> 320 us; 1,792 instances of 8 models 89 -> 50 us.
constexpr int kChunk = 128;          // ticks per chunk

// A row word, from its low bits: receiver, rank (1..MP-1), tick. Words of
// donors compare by tick, then by rank, which is distinct within a tick.
template <class W, int RB> struct RowWordOf {
  using Word = W;
  static constexpr int kRank = RB, kTick = 2 * RB;
  static constexpr uint32_t kRecv = (1u << RB) - 1, kEnd = (uint32_t)kChunk << kTick;
  static constexpr uint32_t kNone = (W)~(W)0;
  static_assert(kEnd < kNone, "the word holds a tick past the chunk");
};
template <int MP> struct RowWord;
template <> struct RowWord<8> : RowWordOf<uint16_t, 3> {};
template <> struct RowWord<16> : RowWordOf<uint16_t, 4> {};
template <> struct RowWord<32> : RowWordOf<uint32_t, 5> {};
template <> struct RowWord<64> : RowWordOf<uint32_t, 6> {};

constexpr uint32_t kNoTick = 0x7f;   // receiver byte of a tick that does nothing
constexpr uint32_t kSlowBit = 0x80;  // receiver byte: the tick rebalances

// order of the values as unsigned keys (-0 equals 0), total also for NaN, so
// that the ranks of a tick are always distinct
__device__ __forceinline__ uint32_t order_key(float z) {
  uint32_t u = __float_as_uint(z);
  if (u == 0x80000000u) u = 0;
  return u ^ ((u >> 31) ? 0xffffffffu : 0x80000000u);
}
__device__ __forceinline__ unsigned long long order_key(double z) {
  unsigned long long u = (unsigned long long)__double_as_longlong(z);
  if (u == 0x8000000000000000ull) u = 0;
  return u ^ ((u >> 63) ? ~0ull : 0x8000000000000000ull);
}

// Position of a donor in its tick's order: group (idle 0, surplus 1, nominal
// 2), Z descending within surplus and nominal, then index; a model that is no
// donor comes after every donor.
template <class T> struct DonorKey;
template <> struct DonorKey<float> {
  unsigned long long k;
  DonorKey() = default;
  __device__ __forceinline__ DonorKey(int g, float z, int m)
      : k(g < 0 ? ~0ull
                : (unsigned long long)g << 38 |
                      (unsigned long long)(g ? ~order_key(z) : 0u) << 6 | (unsigned)m) {}
  __device__ __forceinline__ bool operator<(const DonorKey& o) const { return k < o.k; }
};
template <> struct DonorKey<double> {
  unsigned long long k;
  unsigned long long gm;
  DonorKey() = default;
  __device__ __forceinline__ DonorKey(int g, double z, int m)
      : k(g > 0 ? ~order_key(z) : 0ull), gm((unsigned long long)(g < 0 ? 3 : g) << 6 | (unsigned)m) {}
  __device__ __forceinline__ bool operator<(const DonorKey& o) const {
    const unsigned ga = (unsigned)gm >> 6, gb = (unsigned)o.gm >> 6;
    return ga != gb ? ga < gb : (k != o.k ? k < o.k : (unsigned)gm < (unsigned)o.gm);
  }
};

// donor group of a model of region rg at a tick that acts, -1 = not a donor
template <class T>
__device__ __forceinline__ int donor_group(uint8_t rg, T z, T zr, bool rescue) {
  if (rg == kIdle) return 0;
  if (rg == kSurp) return 1;
  if (rg == kNom && (rescue || z > zr)) return 2;   // rebalance: nominal above the receiver
  return -1;
}

// The chunk a CTA ranks, and the window of its ticks
template <class T> struct ChunkOf {
  int s, ti, c0, nf;
  uint32_t win;
  __device__ __forceinline__ ChunkOf(const WalkBatch<T>& b) {
    s = prefix_index(b.ent_base, b.n_series, blockIdx.x, b.n_tau);
    const int local = (int)(blockIdx.x - (int64_t)b.ent_base[s] * b.n_tau);
    const int nch = b.ent_base[s + 1] - b.ent_base[s];
    ti = local / nch;
    c0 = (local - ti * nch) * kChunk;
    // K * win < 2^31, so every tick time fits 32 unsigned bits
    win = (uint32_t)b.series_win[s];
    nf = (int)((uint32_t)b.series_K[s] * win / (uint32_t)b.fast_ms);
  }
};

// From the ranks (0 = not a donor) and receiver bytes of a chunk's ticks in
// shared memory: the row words, a suffix minimum per column -- each thread
// finds its segment's first donor tick, then writes its segment backwards from
// the first one after it -- and the next tick that does anything.
template <int MP, int THREADS>
__device__ __forceinline__ void write_rows(const uint8_t (*s_rank)[MP], const uint8_t* s_rec,
                                           void* row_words, uint8_t* recs, uint8_t* nexts) {
  using R = RowWord<MP>;
  using Word = typename R::Word;
  constexpr int NSEG = THREADS / MP < 16 ? THREADS / MP : 16, SEGL = kChunk / NSEG;
  __shared__ Word s_first[NSEG][MP];
  auto word = [&](int u, uint32_t r) {
    return (uint32_t)u << R::kTick | r << R::kRank | (s_rec[u] & R::kRecv);
  };
  const int col = threadIdx.x % MP, seg = threadIdx.x / MP;
  if (seg < NSEG) {
    uint32_t f = R::kEnd;
#pragma unroll
    for (int i = SEGL - 1; i >= 0; --i) {
      const uint32_t r = s_rank[seg * SEGL + i][col];
      if (r) f = word(seg * SEGL + i, r);
    }
    s_first[seg][col] = (Word)f;
  }
  __syncthreads();
  const size_t base = (size_t)blockIdx.x * kChunk;
  if (seg < NSEG) {
    uint32_t v = R::kEnd;
#pragma unroll
    for (int j = 1; j < NSEG; ++j)
      if (j > seg) v = min(v, (uint32_t)s_first[j][col]);
    Word* out = static_cast<Word*>(row_words) + base * MP + col;
#pragma unroll
    for (int i = SEGL - 1; i >= 0; --i) {
      const int ul = seg * SEGL + i;
      const uint32_t r = s_rank[ul][col];
      if (r) v = word(ul, r);
      out[(size_t)ul * MP] = (Word)v;
    }
  }
  if (threadIdx.x < kChunk) {
    const int lane = threadIdx.x & 31;
    int nx = kChunk;
    for (int g = kChunk / 32 - 1; g >= (int)threadIdx.x / 32; --g) {
      unsigned on = __ballot_sync(0xffffffffu, s_rec[32 * g + lane] != kNoTick);
      if (g == (int)threadIdx.x / 32) on &= 0xffffffffu << lane;
      if (on) nx = 32 * g + __ffs(on) - 1;
    }
    recs[base + threadIdx.x] = s_rec[threadIdx.x];
    nexts[base + threadIdx.x] = (uint8_t)nx;
  }
}

// Up to 16 models: one CTA per (series, tau, chunk), one thread per tick with
// its row in registers; every pair of models is compared once. Bound by the
// instructions of its few warps (4,320 ticks of 16 models: 12 us; spreading a
// tick's models over lanes and counting from shuffles took 15).
template <class T, int MP, bool QUAD>
__global__ void __launch_bounds__(kChunk)
k_tick_rows(const __grid_constant__ WalkBatch<T> b, void* __restrict__ rows,
            uint8_t* __restrict__ recs, uint8_t* __restrict__ nexts) {
  __shared__ uint8_t s_rank[kChunk][MP];
  __shared__ uint8_t s_rec[kChunk];
  const int M = b.M;
  const ChunkOf<T> ch(b);
  const int u = ch.c0 + threadIdx.x;
  uint32_t rec = kNoTick;
  int rank[MP];
#pragma unroll
  for (int m = 0; m < MP; ++m) rank[m] = 0;
  if (u < ch.nf) {
    // window whose right edge passes the tick
    const uint32_t k =
        FastDiv(ch.win).div((uint32_t)(u + 1) * (uint32_t)b.fast_ms + ch.win - 1u) - 1u;
    const size_t x = (size_t)b.series_off[ch.s] + (size_t)k * M;
    T z[MP];
    uint8_t rg[MP];
#pragma unroll
    for (int m = 0; m < MP; m += 4) {
      if (QUAD && m < M) {
        load_quad(b.Z + x + m, z + m);
        const uchar4 c4 = *reinterpret_cast<const uchar4*>(b.cls + x + m);
        rg[m] = c4.x; rg[m + 1] = c4.y; rg[m + 2] = c4.z; rg[m + 3] = c4.w;
      } else {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          z[m + i] = m + i < M ? b.Z[x + m + i] : (T)0;
          rg[m + i] = m + i < M ? b.cls[x + m + i] : kIdle;
        }
      }
    }
    const bool tau_dev = b.tau_crit != nullptr;
    const T tau_v = b.tau_list[tau_dev ? 0 : ch.ti];
    bool rescue = false;
#pragma unroll
    for (int m = 0; m < MP; ++m)
      if (m < M) {
        rg[m] = region_of(rg[m], z[m], tau_dev ? b.tau_crit[m] : tau_v, b.tau_surp[m]);
        rescue |= rg[m] == kCrit;
      }
    // receiver: rescue -> lowest Z among critical; rebalance -> among non-idle
    const bool slow = (u + 1) % (b.slow_ms / b.fast_ms) == 0;
    int recv = -1;
    T zr = (T)0;
#pragma unroll
    for (int m = 0; m < MP; ++m) {
      const bool cand = m < M && (rescue ? rg[m] == kCrit : slow && rg[m] != kIdle);
      if (cand && (recv < 0 || z[m] < zr)) {
        recv = m;
        zr = z[m];
      }
    }
    if (recv >= 0 && (rescue || zr < (T)1)) {
      rec = (uint32_t)recv | (rescue ? 0u : kSlowBit);
      DonorKey<T> key[MP];
      bool don[MP];
#pragma unroll
      for (int m = 0; m < MP; ++m) {
        const int g = m < M && m != recv ? donor_group(rg[m], z[m], zr, rescue) : -1;
        don[m] = g >= 0;
        key[m] = DonorKey<T>(g, z[m], m);
        rank[m] = 1;
      }
#pragma unroll
      for (int m = 1; m < MP; ++m)
#pragma unroll
        for (int q = 0; q < m; ++q) {
          const bool first = key[q] < key[m];
          rank[m] += first;
          rank[q] += !first;
        }
#pragma unroll
      for (int m = 0; m < MP; ++m) rank[m] = don[m] ? rank[m] : 0;
    }
  }
  s_rec[threadIdx.x] = (uint8_t)rec;
#pragma unroll
  for (int m = 0; m < MP; m += 4)
    *reinterpret_cast<uint32_t*>(&s_rank[threadIdx.x][m]) =
        (uint32_t)rank[m] | (uint32_t)rank[m + 1] << 8 | (uint32_t)rank[m + 2] << 16 |
        (uint32_t)rank[m + 3] << 24;
  __syncthreads();
  write_rows<MP, kChunk>(s_rank, s_rec, rows, recs, nexts);
}

// 17 to 64 models: a warp per tick, models on lanes (two per lane above 32);
// rows of Z and regions are read coalesced and a model's rank is counted
// against the tick's keys in shared memory (64 models, 17,280 ticks: 24 us, at
// 80 % of the issue slots; one thread per model on scattered loads took 202).
constexpr int kWideThreads = 1024;
template <class T, int MP>
__global__ void __launch_bounds__(kWideThreads)
k_tick_rows_wide(const __grid_constant__ WalkBatch<T> b, void* __restrict__ rows,
                 uint8_t* __restrict__ recs, uint8_t* __restrict__ nexts) {
  constexpr int MPL = MP / 32;
  __shared__ uint8_t s_rank[kChunk][MP];
  __shared__ uint8_t s_rec[kChunk];
  __shared__ __align__(16) DonorKey<T> s_key[kWideThreads / 32][MP];
  const unsigned full = 0xffffffffu;
  const int M = b.M;
  const ChunkOf<T> ch(b);
  const FastDiv fwin(ch.win);
  const int ratio = b.slow_ms / b.fast_ms;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const bool tau_dev = b.tau_crit != nullptr;
  T tc[MPL], tsu[MPL];
#pragma unroll
  for (int j = 0; j < MPL; ++j) {
    const int m = lane + 32 * j;
    tc[j] = m < M ? (tau_dev ? b.tau_crit[m] : b.tau_list[ch.ti]) : (T)0;
    tsu[j] = m < M ? b.tau_surp[m] : (T)0;
  }
  for (int ul = warp; ul < kChunk; ul += kWideThreads / 32) {
    const int u = ch.c0 + ul;
    uint32_t rec = kNoTick;
    int rank[MPL];
#pragma unroll
    for (int j = 0; j < MPL; ++j) rank[j] = 0;
    if (u < ch.nf) {
      const uint32_t k = fwin.div((uint32_t)(u + 1) * (uint32_t)b.fast_ms + ch.win - 1u) - 1u;
      const size_t x = (size_t)b.series_off[ch.s] + (size_t)k * M + lane;
      T z[MPL];
      uint8_t rg[MPL];
      unsigned crit[MPL], live[MPL];
      bool rescue = false;
#pragma unroll
      for (int j = 0; j < MPL; ++j) {
        const bool has = lane + 32 * j < M;
        z[j] = has ? b.Z[x + 32 * j] : (T)0;
        rg[j] = has ? region_of(b.cls[x + 32 * j], z[j], tc[j], tsu[j]) : (uint8_t)0xff;
        crit[j] = __ballot_sync(full, rg[j] == kCrit);
        live[j] = __ballot_sync(full, has && rg[j] != kIdle);
        rescue |= crit[j] != 0;
      }
      const bool slow = (u + 1) % ratio == 0;
      // receiver: lowest Z among the candidates, lowest index on ties (a NaN
      // stays only where it is the first candidate, as in an ascending scan)
      int recv = -1;
      T zr = (T)0;
#pragma unroll
      for (int j = 0; j < MPL; ++j) {
        const unsigned cand = rescue ? crit[j] : (slow ? live[j] : 0u);
        if (!cand) continue;
        const unsigned num = cand & ~__ballot_sync(full, z[j] != z[j]);
        int w = __ffs(cand) - 1;
        if (recv >= 0 && !num) continue;
        if (recv >= 0 || (num >> w & 1u)) {
          const auto key = order_key(z[j]);
          const bool in = num >> lane & 1u;
          const uint32_t hi = sizeof(T) == 8 ? (uint32_t)((unsigned long long)key >> 32)
                                             : (uint32_t)key;
          const uint32_t mh = __reduce_min_sync(full, in ? hi : 0xffffffffu);
          bool low = in && hi == mh;
          if (sizeof(T) == 8) {
            const uint32_t ml = __reduce_min_sync(full, low ? (uint32_t)key : 0xffffffffu);
            low = low && (uint32_t)key == ml;
          }
          w = __ffs(__ballot_sync(full, low)) - 1;
        }
        const T zw = __shfl_sync(full, z[j], w);
        if (recv < 0 || zw < zr) {
          recv = w + 32 * j;
          zr = zw;
        }
      }
      if (recv >= 0 && (rescue || zr < (T)1)) {
        rec = (uint32_t)recv | (rescue ? 0u : kSlowBit);
        DonorKey<T> key[MPL];
        bool don[MPL];
#pragma unroll
        for (int j = 0; j < MPL; ++j) {
          const int m = lane + 32 * j;
          const int g = m != recv ? donor_group(rg[j], z[j], zr, rescue) : -1;
          don[j] = g >= 0;
          key[j] = DonorKey<T>(g, z[j], m);
          s_key[warp][m] = key[j];
          rank[j] = 1;
        }
        __syncwarp();
#pragma unroll 16
        for (int q = 0; q < MP; ++q) {
          const DonorKey<T> kq = s_key[warp][q];
#pragma unroll
          for (int j = 0; j < MPL; ++j) rank[j] += kq < key[j];
        }
        __syncwarp();
#pragma unroll
        for (int j = 0; j < MPL; ++j) rank[j] = don[j] ? rank[j] : 0;
      }
    }
    if (lane == 0) s_rec[ul] = (uint8_t)rec;
#pragma unroll
    for (int j = 0; j < MPL; ++j) s_rank[ul][lane + 32 * j] = (uint8_t)rank[j];
  }
  __syncthreads();
  write_rows<MP, kWideThreads>(s_rank, s_rec, rows, recs, nexts);
}

// What the walk reads, by value: per-series tick counts and the controllers.
struct LaneWalk {
  int M, n_tau, n_cap, slab, n_buf;  // slab: ticks staged at a time (a multiple of kChunk)
  int32_t chunk_base[kMaxSeries + 1], win[kMaxSeries], cap_list[kMaxCap];
  int32_t fast_ms;
  int64_t budget, moves_cap;
  const int32_t *r_min, *footprint, *r0;
  int32_t* r_out;
  tre_move* moves;
  int64_t* n_moves;
  tre_diag* diag;
  const void* rows;
  const uint8_t *recs, *nexts;
};

constexpr int kLaneThreads = 256;
constexpr int kLaneLog = 256;      // moves a warp collects before it writes them out
// bytes of one staged tick: its row, receiver and next acting tick; a buffer
// ends in a row of "none", read when a walk steps past the last tick
template <int MP> __host__ __device__ constexpr int slab_bytes(int ticks) {
  return ticks * (MP * (int)sizeof(typename RowWord<MP>::Word) + 2) +
         MP * (int)sizeof(typename RowWord<MP>::Word);
}

__device__ __forceinline__ void copy16(void* smem, const void* gmem) {
  const unsigned sa = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(sa), "l"(gmem) : "memory");
}

// One CTA per (series, tau) and group of kLaneThreads / 32 pacing caps, one
// warp per controller instance. The rows of `slab` ticks are staged in shared
// memory, the next slab's loads in flight while this one is walked. What bounds
// it is the chain of one move: row load, mask, warp minimum, receiver load,
// counts. Moves go to a log in shared memory (tick, position in the tick,
// donor) and are written out by the whole warp, so that nothing in the chain
// branches on a lane (a move with unit footprints and one transition a tick
// takes 200 cycles; writing its record from the donor's lane took 525).
template <int MP>
__global__ void __launch_bounds__(kLaneThreads)
k_walk_lane(const __grid_constant__ LaneWalk w) {
  extern __shared__ __align__(16) unsigned char dyn[];
  __shared__ uint32_t s_log[kLaneThreads / 32][kLaneLog];
  __shared__ int s_foot[64];
  constexpr int MPL = MP > 32 ? 2 : 1, L1 = MPL - 1;
  using R = RowWord<MP>;
  using Word = typename R::Word;
  constexpr uint32_t kNone = R::kNone;
  const unsigned full = 0xffffffffu;
  const int ti = blockIdx.x % w.n_tau, si = blockIdx.x / w.n_tau;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int ci = blockIdx.y * (kLaneThreads / 32) + warp;
  const int M = w.M;
  const int nch = w.chunk_base[si + 1] - w.chunk_base[si];
  const int n_tick = nch * kChunk;                  // the last chunk's padding does nothing
  const size_t t0 = ((size_t)w.chunk_base[si] * w.n_tau + (size_t)ti * nch) * kChunk;
  const int buf_bytes = slab_bytes<MP>(w.slab);
  // a buffer: rows [slab + 1][MP] words, receiver bytes, next-tick bytes
  auto fetch = [&](int first, int buf) {
    const int n = min(w.slab, n_tick - first);
    unsigned char* d = dyn + buf * buf_bytes;
    const unsigned char* src =
        reinterpret_cast<const unsigned char*>(static_cast<const Word*>(w.rows) + (t0 + first) * MP);
    for (int i = threadIdx.x; i < n * MP * (int)sizeof(Word) / 16; i += kLaneThreads)
      copy16(d + 16 * i, src + 16 * i);
    if (threadIdx.x < MP) reinterpret_cast<Word*>(d)[n * MP + threadIdx.x] = (Word)R::kEnd;
    d += (size_t)(w.slab + 1) * MP * sizeof(Word);
    for (int i = threadIdx.x; i < n / 16; i += kLaneThreads) {
      copy16(d + 16 * i, w.recs + t0 + first + 16 * i);
      copy16(d + w.slab + 16 * i, w.nexts + t0 + first + 16 * i);
    }
  };
  if (n_tick > 0) fetch(0, 0);
  asm volatile("cp.async.commit_group;\n" ::: "memory");
  if (threadIdx.x < M) s_foot[threadIdx.x] = w.footprint[threadIdx.x];   // read past the slab's barrier

  // the instance's state: replicas above the floor per model, the idle pool
  const bool mine = ci < w.n_cap;
  const int inst = (si * w.n_tau + ti) * w.n_cap + (mine ? ci : 0);
  const int Kp = mine ? w.cap_list[ci] : 0;
  const int64_t cap = w.moves_cap;
  tre_move* mv = w.moves + (size_t)inst * cap;
  int c[MPL], rmin[MPL], g[MPL];
  int64_t pool = 0;
  bool bad = false, unit = true;
#pragma unroll
  for (int j = 0; j < MPL; ++j) {
    const int m = lane + 32 * j;
    c[j] = rmin[j] = 0;
    g[j] = 1;
    if (mine && m < M) {
      const int r = w.r0[m];
      rmin[j] = w.r_min[m];
      g[j] = w.footprint[m];
      pool += (int64_t)g[j] * r;
      bad |= r < 0 || g[j] < 1 || rmin[j] < 0;
      unit &= g[j] == 1;
      c[j] = r - rmin[j];
    }
  }
  for (int o = 16; o > 0; o >>= 1) pool += __shfl_xor_sync(full, pool, o);
  pool = w.budget - pool;
  // an inconsistent controller state (negative replicas or floors, footprint
  // below one, replicas beyond the budget) produces no moves
  bad = __any_sync(full, bad) || pool < 0;
  unit = __all_sync(full, unit);
  const bool walks = mine && !bad && Kp > 0;
  const FastDiv fwin((uint32_t)w.win[si]);
  uint32_t* log = s_log[warp];
  int64_t n_out = 0;   // moves written out
  int n_log = 0;       // moves in the log: tick | position << 11 | donor << 19 (64: the pool)

  // a slab of n ticks, the first of them tick `first` of the series
  auto walk = [&](const Word* rows, const uint8_t* recs, const uint8_t* nexts, int n,
                  int first) {
    const Word* my = rows + (lane & (MP - 1));
    // all ones where the model has nothing above its floor
    uint32_t no[MPL];
    auto masks = [&]() {
#pragma unroll
      for (int j = 0; j < MPL; ++j) no[j] = c[j] > 0 ? 0u : kNone;
    };
    masks();
    auto flush = [&]() {
      __syncwarp();
      for (int i = lane; i < n_log; i += 32) {
        const uint32_t e = log[i];
        const int a = e & 2047u, d = (int)(e >> 19);
        const uint32_t rec = recs[a];
        put_move(mv, n_out + i, cap,
                 (int32_t)fwin.div((uint32_t)(first + a + 1) * (uint32_t)w.fast_ms +
                                   (uint32_t)w.win[si] - 1u) - 1,
                 (int)(rec & 63u), d == 64 ? -1 : d,
                 rec & kSlowBit ? TRE_REBALANCE : TRE_RESCUE, (int)(e >> 11 & 255u));
      }
      __syncwarp();
      n_out += n_log;
      n_log = 0;
    };
    // between two appends the log is never full: either one flushes it before or as
    // it fills (a run is at most 255 moves, so an empty log takes any)
    auto log_one = [&](bool here, uint32_t a, int seq, int donor) {
      if (here) log[n_log] = a | (uint32_t)seq << 11 | (uint32_t)donor << 19;
      if (++n_log == kLaneLog) flush();
    };
    auto log_run = [&](uint32_t a, int seq, int donor, int take) {   // take <= 255
      if (n_log + take >= kLaneLog) flush();
      for (int q = lane; q < take; q += 32)
        log[n_log + q] = a | (uint32_t)(seq + q) << 11 | (uint32_t)donor << 19;
      n_log += take;
    };
    auto receive = [&](int recv, int take) {
      c[0] += lane == recv ? take : 0;
      if (MPL > 1) c[L1] += lane + 32 == recv ? take : 0;
    };
    int u = 0;
    int left = Kp;      // transitions the tick at u may still make
    if (unit) {
      // the idle pool first: it only shrinks, and every acting tick draws on it
      while (pool > 0 && u < n) {
        const int a = (u & ~(kChunk - 1)) + nexts[u];
        if (nexts[u] == kChunk) {
          u = a;
          continue;
        }
        const int take = pool < Kp ? (int)pool : Kp;
        pool -= take;
        log_run((uint32_t)a, 0, 64, take);
        receive(recs[a] & 63, take);
        left = Kp - take;
        u = left > 0 ? a : a + 1;
        if (left == 0) left = Kp;
      }
      masks();
      if (u >= n) {
        flush();
        return;
      }
    }
    if (unit && Kp == 1) {
      // one replica per tick: every tick found moves exactly one
      while (true) {
        const uint32_t k0 = my[u * MP] | no[0];
        const uint32_t k1 = MPL > 1 ? my[u * MP + 32] | no[L1] : kNone;
        const uint32_t best = __reduce_min_sync(full, MPL > 1 ? min(k0, k1) : k0);
        const int t = (int)(best >> R::kTick), cb = u & ~(kChunk - 1);
        if (t >= kChunk) {                      // nothing in the rest of the chunk
          u = cb + kChunk;
          if (u >= n) break;
          continue;
        }
        const int a = cb + t;
        const int recv = (int)(best & R::kRecv);
        const bool d0 = k0 == best, d1 = MPL > 1 && k1 == best;
        c[0] += (lane == recv) - d0;
        if (MPL > 1) c[L1] += (lane + 32 == recv) - d1;
        masks();
        log_one(d0 || d1, (uint32_t)a, 0, lane + (d1 ? 32 : 0));
        u = a + 1;
      }
    } else if (unit) {
      // up to Kp replicas per tick: donors in rank order, each giving what it
      // has above its floor
      int cur = u;
      while (true) {
        const uint32_t k0 = my[u * MP] | no[0];
        const uint32_t k1 = MPL > 1 ? my[u * MP + 32] | no[L1] : kNone;
        const uint32_t best = __reduce_min_sync(full, MPL > 1 ? min(k0, k1) : k0);
        const int t = (int)(best >> R::kTick), cb = u & ~(kChunk - 1);
        if (t >= kChunk) {
          u = cb + kChunk;
          if (u >= n) break;
          continue;
        }
        const int a = cb + t;
        if (a != cur) {
          cur = a;
          left = Kp;
        }
        const int recv = (int)(best & R::kRecv);
        const bool d0 = k0 == best, d1 = MPL > 1 && k1 == best;
        const int give = min(d1 ? c[L1] : c[0], left);
        const int take = (int)__reduce_max_sync(full, d0 || d1 ? (unsigned)give : 0u);
        if (d0) c[0] -= take;
        if (MPL > 1 && d1) c[L1] -= take;
        receive(recv, take);
        masks();
        const int src = __ffs(__ballot_sync(full, d0 || d1)) - 1;   // ranks are distinct
        const unsigned up = MPL > 1 ? __ballot_sync(full, d1) : 0u;
        log_run((uint32_t)a, Kp - left, src + (up ? 32 : 0), take);
        left -= take;
        u = left > 0 ? a : a + 1;
      }
    } else {
      // footprints differ: per transition the pool if it covers the receiver's
      // footprint, else donor replicas until it is covered; an uncoverable
      // transition releases nothing and ends the tick
      while (true) {
        uint32_t k = my[u * MP] | no[0];
        if (MPL > 1) k = min(k, my[u * MP + 32] | no[L1]);
        const uint32_t next = __reduce_min_sync(full, k);
        const int cb = u & ~(kChunk - 1);
        int t = (int)(next >> R::kTick), recv = (int)(next & R::kRecv);
        if (pool > 0 && u < n && (int)nexts[u] < t) {
          t = nexts[u];
          recv = recs[cb + t] & 63;
        }
        if (t >= kChunk) {
          u = cb + kChunk;
          if (u >= n) break;
          continue;
        }
        const int a = cb + t;
        const int need = s_foot[recv];
        // the donors of this very tick, from the words of the row at the tick
        // itself: rank above, footprint below (65,535 and more: looked up), so
        // that one warp minimum finds the next donor and what it frees
        uint32_t q[MPL];
#pragma unroll
        for (int j = 0; j < MPL; ++j) {
          const uint32_t r = my[a * MP + 32 * j];
          q[j] = (int)(r >> R::kTick) == t
                     ? (r >> R::kRank & R::kRecv) << 16 | (uint32_t)min(g[j], 0xffff)
                     : ~0u;
        }
        for (int seq = 0; seq < Kp; ++seq) {
          if (pool >= need) {
            pool -= need;
            log_one(lane == 0, (uint32_t)a, seq, 64);
            receive(recv, 1);
            continue;
          }
          int64_t f = pool;
          const int64_t n0 = n_out + n_log;
          int h[MPL];
#pragma unroll
          for (int j = 0; j < MPL; ++j) h[j] = c[j];
          while (f < need) {
            const uint32_t e0 = h[0] > 0 ? q[0] : ~0u;
            const uint32_t e1 = MPL > 1 && h[L1] > 0 ? q[L1] : ~0u;
            const uint32_t best = __reduce_min_sync(full, MPL > 1 ? min(e0, e1) : e0);
            if (best == ~0u) break;
            const bool d0 = e0 == best, d1 = MPL > 1 && e1 == best;
            uint32_t frees = best & 0xffffu;
            if (frees == 0xffffu)
              frees = __reduce_max_sync(full, d0 ? (unsigned)g[0] : d1 ? (unsigned)g[L1] : 0u);
            f += frees;
            h[0] -= d0;
            if (MPL > 1) h[L1] -= d1;
            log_one(d0 || d1, (uint32_t)a, seq, lane + (d1 ? 32 : 0));
          }
          if (f < need) {                       // take the tentative releases back
            if (n0 < n_out) {
              n_out = n0;
              n_log = 0;
            } else {
              n_log = (int)(n0 - n_out);
            }
            break;
          }
#pragma unroll
          for (int j = 0; j < MPL; ++j) c[j] = h[j];
          pool = f - need;
          receive(recv, 1);
        }
        masks();
        u = a + 1;
      }
    }
    flush();
  };

  int buf = 0;
  for (int first = 0; first < n_tick; first += w.slab, buf ^= w.n_buf - 1) {
    const int more = first + w.slab;
    if (more < n_tick) fetch(more, buf ^ 1);
    asm volatile("cp.async.commit_group;\n" ::: "memory");
    asm volatile("cp.async.wait_group 1;\n" ::: "memory");
    __syncthreads();
    const unsigned char* d = dyn + buf * buf_bytes;
    const uint8_t* recs = d + (size_t)(w.slab + 1) * MP * sizeof(Word);
    if (walks)
      walk(reinterpret_cast<const Word*>(d), recs, recs + w.slab, min(w.slab, n_tick - first),
           first);
    __syncthreads();
  }
  if (!mine) return;
#pragma unroll
  for (int j = 0; j < MPL; ++j) {
    const int m = lane + 32 * j;
    if (m < M) w.r_out[(size_t)inst * M + m] = c[j] + rmin[j];
  }
  if (lane == 0) {
    w.n_moves[inst] = n_out;
    if (bad) w.diag->err = TRE_EINVAL;
    else if (n_out > cap) w.diag->err = TRE_EOVERFLOW;
  }
}

constexpr size_t kStageMax = 160 * 1024;

template <class T, int MPL>
cudaError_t walk_launch(const WalkBatch<T>& b, WalkWs& w, cudaStream_t s) {
  int max_ent = 0;
  for (int i = 0; i < b.n_series; ++i) max_ent = std::max(max_ent, b.ent_base[i + 1] - b.ent_base[i]);
  const size_t smem = 2 * (((size_t)max_ent * 2 + 15) & ~(size_t)15) +
                      2 * (((size_t)max_ent * b.M * 2 + 15) & ~(size_t)15);
  const dim3 grid((unsigned)(b.n_series * b.n_tau),
                  (unsigned)((b.n_cap + kCapWarps - 1) / kCapWarps));
  const unsigned th = (unsigned)(std::min(b.n_cap, kCapWarps) * 32);
  if (smem <= kStageMax) {
    cudaError_t e = func_smem_once((const void*)k_walk<T, MPL, true>, (int)kStageMax, false);
    if (e) return e;
    k_walk<T, MPL, true><<<grid, th, smem, s>>>(b, w.recv, w.n_donor, w.rank, w.order, w.dm64);
  } else {
    k_walk<T, MPL, false><<<grid, th, 0, s>>>(b, w.recv, w.n_donor, w.rank, w.order, w.dm64);
  }
  return cudaGetLastError();
}

// The lane walk takes nested cadences (every slow tick a fast tick, no fast
// tick shorter than a window, so a window ends at most one tick) and up to 64
// models (two per lane; a row word has six rank bits). Elsewhere ticks are
// visited one by one.
template <class T> bool lane_walk(const WalkBatch<T>& b) {
  if (b.M > 64 || b.slow_ms % b.fast_ms != 0) return false;
  for (int s = 0; s < b.n_series; ++s)
    if (b.fast_ms < b.series_win[s]) return false;
  return true;
}

int row_models(int M) { return M <= 8 ? 8 : M <= 16 ? 16 : M <= 32 ? 32 : 64; }

template <class T, int MP>
cudaError_t lane_launch(const WalkBatch<T>& b, const WalkWs& w, cudaStream_t s, int* launches) {
  const int64_t chunks = (int64_t)b.ent_base[b.n_series] * b.n_tau;
  if (chunks > 0) {
    if constexpr (MP <= 16) {
      // rows start on 16-byte boundaries when M is a multiple of 4 (series
      // offsets are multiples of M) and both arrays are 16-byte aligned
      if (b.M % 4 == 0 && (((uintptr_t)b.Z | (uintptr_t)b.cls) & 15) == 0)
        k_tick_rows<T, MP, true><<<(unsigned)chunks, kChunk, 0, s>>>(b, w.rows, w.recs, w.nexts);
      else
        k_tick_rows<T, MP, false><<<(unsigned)chunks, kChunk, 0, s>>>(b, w.rows, w.recs, w.nexts);
    } else {
      k_tick_rows_wide<T, MP><<<(unsigned)chunks, kWideThreads, 0, s>>>(b, w.rows, w.recs,
                                                                        w.nexts);
    }
    if (launches) ++*launches;
  }
  LaneWalk v;
  v.M = b.M;
  v.n_tau = b.n_tau;
  v.n_cap = b.n_cap;
  int longest = 0;
  for (int i = 0; i < b.n_series; ++i) {
    v.chunk_base[i] = b.ent_base[i];
    v.win[i] = b.series_win[i];
    longest = std::max(longest, (b.ent_base[i + 1] - b.ent_base[i]) * kChunk);
  }
  v.chunk_base[b.n_series] = b.ent_base[b.n_series];
  for (int i = 0; i < b.n_cap; ++i) v.cap_list[i] = b.cap_list[i];
  v.fast_ms = b.fast_ms;
  v.budget = b.budget;
  v.moves_cap = b.moves_cap;
  v.r_min = b.r_min;
  v.footprint = b.footprint;
  v.r0 = b.r0;
  v.r_out = b.r_out;
  v.moves = b.moves;
  v.n_moves = b.n_moves;
  v.diag = b.diag;
  v.rows = w.rows;
  v.recs = w.recs;
  v.nexts = w.nexts;
  // short series are staged whole; longer ones in two buffers, the next
  // slab's load behind the walk of this one
  constexpr int kSlab = MP == 64 ? 384 : MP == 32 ? 768 : 1024;
  constexpr int kSmem = 2 * slab_bytes<MP>(kSlab);
  static_assert(kSmem <= 200 * 1024, "two slabs and the logs fit a block's shared memory");
  static_assert(kSlab < 2048, "a logged tick has 11 bits");
  v.slab = longest <= kSlab ? std::max(longest, kChunk) : kSlab;
  v.n_buf = longest <= kSlab ? 1 : 2;
  cudaError_t e = func_smem_once((const void*)k_walk_lane<MP>, kSmem, false);
  if (e) return e;
  const dim3 grid((unsigned)(b.n_series * b.n_tau),
                  (unsigned)((b.n_cap + kLaneThreads / 32 - 1) / (kLaneThreads / 32)));
  k_walk_lane<MP><<<grid, kLaneThreads, (size_t)slab_bytes<MP>(v.slab) * v.n_buf, s>>>(v);
  if (launches) ++*launches;
  return cudaGetLastError();
}

template <class T, int MMAX>
cudaError_t walk_thread_launch(const WalkBatch<T>& b, WalkWs& w, size_t smem, cudaStream_t s) {
  cudaError_t e = func_smem_once((const void*)k_walk_thread<T, MMAX>, (int)kStageMax, false);
  if (e) return e;
  k_walk_thread<T, MMAX><<<b.n_series * b.n_tau, 32, smem, s>>>(b, w.recv, w.packed, w.dmask);
  return cudaGetLastError();
}

}  // namespace

template <class T> void walk_ws_layout(Arena& a, WalkBatch<T>& b, WalkWs& w) {
  w = WalkWs{};
  const bool lanes = lane_walk(b);
  // entries per series: chunks of fast ticks (lane walk), else its fast and
  // its slow ticks
  int64_t total = 0;
  for (int s = 0; s < b.n_series; ++s) {
    b.ent_base[s] = (int32_t)total;
    const int64_t span = (int64_t)b.series_K[s] * b.series_win[s];
    total += lanes ? (span / b.fast_ms + kChunk - 1) / kChunk
                   : span / b.fast_ms + span / b.slow_ms;
  }
  b.ent_base[b.n_series] = (int32_t)total;
  const size_t ents = (size_t)std::max<int64_t>(total * b.n_tau, 1);
  if (lanes) {
    const int words = row_models(b.M);
    w.rows = a.take<uint32_t>(ents * kChunk * words / (words <= 16 ? 2 : 1));
    w.recs = a.take<uint8_t>(ents * kChunk);
    w.nexts = a.take<uint8_t>(ents * kChunk);
    return;
  }
  w.recv = a.take<int16_t>(ents);
  w.n_donor = a.take<int16_t>(ents);
  w.rank = a.take<uint16_t>(ents * b.M);
  w.order = a.take<uint16_t>(ents * b.M);
  w.packed = a.take<unsigned long long>(ents);
  w.dmask = a.take<uint32_t>(ents);
  w.dm64 = a.take<unsigned long long>(ents);
}

template <class T>
cudaError_t launch_walk(const WalkBatch<T>& b, WalkWs& w, cudaStream_t s, int* launches) {
  if (launches) *launches = 0;
  if (b.n_inst == 0) return cudaSuccess;
  if (lane_walk(b)) {
    switch (row_models(b.M)) {
      case 8: return lane_launch<T, 8>(b, w, s, launches);
      case 16: return lane_launch<T, 16>(b, w, s, launches);
      case 32: return lane_launch<T, 32>(b, w, s, launches);
      default: return lane_launch<T, 64>(b, w, s, launches);
    }
  }
  const int64_t ents = (int64_t)b.ent_base[b.n_series] * b.n_tau;
  // which walk runs decides whether the per-model rank tables are needed
  int max_ent = 0;
  for (int i = 0; i < b.n_series; ++i)
    max_ent = std::max(max_ent, b.ent_base[i + 1] - b.ent_base[i]);
  const size_t thread_smem = (size_t)max_ent * (8 + 4 + 2) + 16;
  const bool thread_walk = b.M <= 16 && b.n_cap <= 32 && thread_smem <= kStageMax;
  // the tick ranking, then the walk
  if (launches) *launches = (ents > 0 ? 1 : 0) + 1;
  if (ents > 0) {
    const unsigned g = (unsigned)((ents + 127) / 128);
    if (b.M <= 8) {
      k_tick_rank_small<T, 8><<<g, 128, 0, s>>>(b, w.recv, w.n_donor, w.rank, w.order, w.packed,
                                                w.dmask, !thread_walk, w.dm64);
    } else if (b.M <= 16) {
      k_tick_rank_small<T, 16><<<g, 128, 0, s>>>(b, w.recv, w.n_donor, w.rank, w.order,
                                                 w.packed, w.dmask, !thread_walk, w.dm64);
    } else if (b.M <= 32) {
      k_tick_rank_small<T, 32><<<g, 128, 0, s>>>(b, w.recv, w.n_donor, w.rank, w.order,
                                                 w.packed, w.dmask, true, w.dm64);
    } else {
      const int64_t th = ents * b.M;
      k_tick_rank<T><<<(unsigned)((th + 255) / 256), 256, 0, s>>>(b, w.recv, w.n_donor, w.rank,
                                                                   w.order, w.dm64);
    }
  }
  if (thread_walk)
    return b.M <= 8 ? walk_thread_launch<T, 8>(b, w, thread_smem, s)
                    : walk_thread_launch<T, 16>(b, w, thread_smem, s);
  const int mpl = (b.M + 31) / 32;
  if (mpl <= 1) return walk_launch<T, 1>(b, w, s);
  if (mpl <= 2) return walk_launch<T, 2>(b, w, s);
  if (mpl <= 4) return walk_launch<T, 4>(b, w, s);
  if (mpl <= 8) return walk_launch<T, 8>(b, w, s);
  if (mpl <= 16) return walk_launch<T, 16>(b, w, s);
  return walk_launch<T, 32>(b, w, s);
}

template void walk_ws_layout<float>(Arena&, WalkBatch<float>&, WalkWs&);
template void walk_ws_layout<double>(Arena&, WalkBatch<double>&, WalkWs&);
template cudaError_t launch_walk<float>(const WalkBatch<float>&, WalkWs&, cudaStream_t, int*);
template cudaError_t launch_walk<double>(const WalkBatch<double>&, WalkWs&, cudaStream_t, int*);

}  // namespace tre
