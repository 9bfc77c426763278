// Resident check periods (see resident.hpp).
//
// What bounds an attempt of a small problem is a chain of latencies: a
// dependent FP64 operation 55-65 cycles, a division 610, a lane sum 405, an L2
// load 350-420, a GPU-scope fence or release 830-880, and the instruction
// fetches of code that each warp runs once per attempt.  So no grid barrier and
// no fence stands between the phases: every element of x+ and y+ that other
// CTAs gather is one word of the value and the number of its attempt (128 bits
// in FP64, 64 in FP32, read and written whole), and a gather that finds an
// older number reads again.  A random gather moves a 32-byte sector either way.
// The sums over the CTAs travel the same way.
//
// Measured (64 attempts with their two checks, reset and result, FP64, against
// the two-kernel path): 4,001 x 10,003 with 60k nonzeros 1,368 -> 700 us; 1,003
// x 8,005 with 376k nonzeros in rows of up to 3,000: 1,918 -> 946 us (1,112 with
// rows of more than 2,048 entries summed by a whole CTA instead of in segments of
// 512 by warps of all CTAs); 50,000 x 200,000 transportation, 400k nonzeros:
// 1,875 -> 1,262 us; 200 x 500 with 2.5k nonzeros, 256 attempts in one CTA: 4,235
// -> 1,815 us.
#include "resident.hpp"

#include <algorithm>
#include <cstddef>
#include <memory>
#include <mutex>

#include "ops.cuh"
#include "resident_sums.cuh"

namespace lpop {

namespace {

constexpr int kStartSpins = 1 << 21;  // polls (~0.3 us each) before a launch gives up on its CTAs all being there
constexpr int kSpins = 1 << 23;       // ... and before a wait for another CTA's word gives up

// The checked build takes both limits from the plan, with an arrival or a word
// that never comes, so that a test can let a wait run out.
#ifdef LPOP_CHECK_BOUNDS
__device__ __forceinline__ int start_spins(const ResPlan& pl) { return pl.test.start_spins ? pl.test.start_spins : kStartSpins; }
__device__ __forceinline__ int wait_spins(const ResPlan& pl) { return pl.test.spins ? pl.test.spins : kSpins; }
__device__ __forceinline__ unsigned int missing_arrivals(const ResPlan& pl) { return (unsigned int)pl.test.missing_arrivals; }
__device__ __forceinline__ unsigned int missing_words(const ResPlan& pl) { return (unsigned int)pl.test.missing_words; }
#else
__device__ __forceinline__ constexpr int start_spins(const ResPlan&) { return kStartSpins; }
__device__ __forceinline__ constexpr int wait_spins(const ResPlan&) { return kSpins; }
__device__ __forceinline__ constexpr unsigned int missing_arrivals(const ResPlan&) { return 0u; }
__device__ __forceinline__ constexpr unsigned int missing_words(const ResPlan&) { return 0u; }
#endif

// The same for a row of more than kBlockRowThreshold entries in FP32: pieces of
// eight terms in FP32, added in FP64, as the step kernels sum such a row.  Only
// one CTA has such a row in one piece (several cut it into segments); a lane has
// up to 110 terms of it.  One FP32 chain of 94 equal terms was off by up to 22 x
// 2^-24 of their sum, the pieces are by less than 2 x 2^-24.  (4 x 2,500 with a
// full row, 256 attempts in the FP32 phase: 2,122 us with the chain, 1,986 so.)
template <int kKind>
__device__ __noinline__ double res_dot_pieces(const float* v, const int* c, int count, int most,
                                              const ResGather<float, kKind>& g) {
  double a = 0.0;
#pragma unroll 1
  for (int k0 = 0; k0 < most; k0 += 8) {
    float p = 0.f;
#pragma unroll
    for (int h = 0; h < 8; h += 4) {
      float xv[4];
      g.four(c, 32, count - k0 - h, xv);
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (k0 + h + u < count) p = fma(v[32 * u], xv[u], p);
      v += 4 * 32;
      c += 4 * 32;
    }
    a += (double)p;
  }
  return a;
}

__device__ __forceinline__ void bar_arrive(unsigned int* bar) {
  asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(bar) : "memory");
}

// Waits until the arrival count has reached `target`; false after `limit` polls.
__device__ __forceinline__ bool bar_wait(const unsigned int* bar, unsigned int target, int limit) {
  for (int k = 0; k < limit; ++k) {
    unsigned int v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(bar) : "memory");
    if ((int)(v - target) >= 0) return true;
  }
  return false;
}

// Sum over the CTAs of one field's records of this attempt (all lanes of the
// calling warp); false when they did not all come.
__device__ __forceinline__ bool rec_sum(const ulonglong2* rec, int G, unsigned int seq, int spins, double* out) {
  const int lane = threadIdx.x & 31;
  constexpr int K = kResMaxCtas / 32;
  double v[K];
  bool done = false;
  for (int k = 0; k < spins && !done; ++k) {
    bool mine = true;
#pragma unroll
    for (int q = 0; q < K; ++q) {
      const int g = lane + 32 * q;
      v[q] = 0.0;
      if (g < G) mine = ResElt<double>::get(rec + g, seq, v + q) && mine;
    }
    done = __all_sync(0xffffffffu, mine);
  }
  static_assert(K == 5, "five records a lane");
  *out = lane_sum(((v[0] + v[1]) + (v[2] + v[3])) + v[4]);
  return done;
}

constexpr int kFacs = 64;
constexpr int kCtlWarps = 3;  // warps that sum the records (a field each); warp 0 then runs the step control

// Barriers of the control warps and of the others.
__device__ __forceinline__ void rows_sync() { asm volatile("bar.sync 2, %0;" ::"n"(kResThreads - 32 * kCtlWarps) : "memory"); }
__device__ __forceinline__ void control_sync() { asm volatile("bar.sync 1, %0;" ::"n"(32 * kCtlWarps) : "memory"); }

// The step scalars that the rows read, as eight words of a broadcast line:
// CTA 0 alone sums the records and runs the step control (every CTA polling
// every record took 2.4 us an attempt with 123 CTAs, mostly queueing at L2).
__device__ __forceinline__ double bcast_word(const DevState& s, int k) {
  switch (k) {
    case 0: return s.eta;
    case 1: return s.step_p;
    case 2: return s.step_d;
    case 3: return s.up_scale_p;
    case 4: return s.up_scale_d;
    case 5: return s.sqrt_gp;
    case 6: return s.sqrt_gd;
    default:
      return __longlong_as_double((long long)s.cur | (long long)s.collect << 1 | (long long)s.pend_p << 2 |
                                  (long long)s.pend_d << 3 | (long long)s.last_accept << 4);
  }
}
__device__ __forceinline__ void bcast_read(DevState& s, int k, double w) {
  switch (k) {
    case 0: s.eta = w; break;
    case 1: s.step_p = w; break;
    case 2: s.step_d = w; break;
    case 3: s.up_scale_p = w; break;
    case 4: s.up_scale_d = w; break;
    case 5: s.sqrt_gp = w; break;
    case 6: s.sqrt_gd = w; break;
    default: {
      const int f = (int)__double_as_longlong(w);
      s.cur = f & 1;
      s.collect = f >> 1 & 1;
      s.pend_p = f >> 2 & 1;
      s.pend_d = f >> 3 & 1;
      s.last_accept = f >> 4 & 1;
    }
  }
}

// kSolo: one CTA, local rows numbered as the global ones, no other CTA to wait for.
//
// One attempt (A^T y of the current y is already in the sums of half cur):
//   rows of A^T: x+ from the sums;
//   rows of A:   A x+ and y+, block sums;
//   warps 0-2:   the CTA's records out; in CTA 0 every CTA's records in,
//                totals, the step control and its result out to the others;
//   the others:  A^T y+ into the sums of half cur ^ 1, which is the next
//                attempt's product if this one is accepted (if not, half cur
//                still holds it); then the averages' terms of the attempt before.
// With words (see resident_kind), nothing is overwritten that another CTA still
// reads: a CTA writes x+ of attempt a + 1 after it has the result of the step
// control, which has every record of attempt a, which its sender wrote
// after its last gather of x+ of attempt a; y+ of attempt a + 1 goes into the
// other half if attempt a was accepted (its last readers finished before the
// records of attempt a), and if it was not, a CTA still reading y+ of attempt
// a takes the newer word for a sum that it will not use.
template <class V, int kKind>
__global__ void __launch_bounds__(kResThreads, 1) resident_kernel(Dev d, Params prm, ResPlan pl, int attempts) {
  constexpr bool kSolo = kKind == kSoloKind, kWords = kKind == kWordsKind, kBars = kKind == kBarriersKind;
  extern __shared__ __align__(16) unsigned char s_raw[];
  __shared__ __align__(16) DevState s_st;
  __shared__ double s_tot[8];
  __shared__ double s_fac[2][kFacs];  // step-size factors of the next kFacs attempts
  __shared__ int s_ok;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const ResLayout L = res_layout(pl, (int)sizeof(V));
  const ResCta C = pl.cta[blockIdx.x];
  const int np = C.p1 - C.p0, nd = C.d1 - C.d0;
  V* const s_vp = reinterpret_cast<V*>(s_raw + L.vp);
  V* const s_vd = reinterpret_cast<V*>(s_raw + L.vd);
  V* const s_xp = reinterpret_cast<V*>(s_raw + L.xp);
  V* const s_xd = reinterpret_cast<V*>(s_raw + L.xd);
  double* const s_red = reinterpret_cast<double*>(s_raw + L.red);
  int* const s_cp = reinterpret_cast<int*>(s_raw + L.cp);
  int* const s_cd = reinterpret_cast<int*>(s_raw + L.cd);
  int2* const s_lrp = reinterpret_cast<int2*>(s_raw + L.lrp);  // first entry, length
  int* const s_gp = reinterpret_cast<int*>(s_raw + L.gp);
  int* const s_gd = reinterpret_cast<int*>(s_raw + L.gd);
  ResItem* const s_it = reinterpret_cast<ResItem*>(s_raw + L.it);
  uint8_t* const s_sense = s_raw + L.sense;
  uint8_t* const s_lenp = s_raw + L.lenp;
  uint8_t* const s_lend = s_raw + L.lend;
  // A^T rows: c l u T 1/T x x xbar sum sum; A rows: b S 1/S y y ybar ax ax
  V* const pc = s_xp;
  V* const plo = pc + pl.rp;
  V* const pup = plo + pl.rp;
  V* const pT = pup + pl.rp;
  V* const piT = pT + pl.rp;
  V* const px = piT + pl.rp;  // two halves
  V* const pxb = px + 2 * pl.rp;
  V* const psum = pxb + pl.rp;  // two halves
  V* const db = s_xd;
  V* const dS = db + pl.rd;
  V* const diS = dS + pl.rd;
  V* const dy_ = diS + pl.rd;  // two halves
  V* const dyb = dy_ + 2 * pl.rd;
  V* const dax = dyb + pl.rd;  // two halves
  const Vecs<V>& v = vecs<V>(d);

  // ---- load the CTA's rows -------------------------------------------------
  {
    const int* src = reinterpret_cast<const int*>(pl.items);
    int* dst = reinterpret_cast<int*>(s_it);
    constexpr int W = sizeof(ResItem) / 4;
#pragma unroll 1
    for (int t = tid; t < np * W; t += kResThreads) dst[t] = src[(size_t)C.p0 * W + t];
#pragma unroll 1
    for (int t = tid; t < nd * W; t += kResThreads) dst[np * W + t] = src[(size_t)C.d0 * W + t];
    const double* ss = reinterpret_cast<const double*>(d.st);
    double* sd = reinterpret_cast<double*>(&s_st);
    for (int t = tid; t < (int)(sizeof(DevState) / 8); t += kResThreads) sd[t] = ss[t];
  }
  __syncthreads();
  const unsigned int base = kSolo ? 0u : pl.bar[1], arrived = kSolo ? 0u : pl.bar[3];
  using Elt = ResElt<V>;
  typename Elt::T* const gxw = reinterpret_cast<typename Elt::T*>(pl.gx);  // [n], then y: [2][m]
  typename Elt::T* const gyw = gxw + d.n;
  {
    const int cur = s_st.cur;
#pragma unroll 1
    for (int i = warp; i < np + nd; i += kResWarps) {
      const bool P = i < np;
      const ResItem I = s_it[i];
      const CsrT<V> M = P ? csr_at<V>(d) : csr_a<V>(d);
      V* sv = (P ? s_vp : s_vd) + I.ent;
      int* sc = (P ? s_cp : s_cd) + I.ent;
      const bool far = kBars && (pl.far >> (P ? 0 : 1) & 1);
      if (I.kind == 0) {  // entry k of the slice's row t at 32 k + t
        if (lane < I.nrows) {
          const int e0 = M.rp[I.row0 + lane], len = M.rp[I.row0 + lane + 1] - e0;
          (P ? s_lenp : s_lend)[I.vec + lane] = (uint8_t)len;
#pragma unroll 4
          for (int k = 0; k < len; ++k) {
            sc[32 * k + lane] = M.ci[e0 + k];
            sv[32 * k + lane] = M.v[e0 + k];
          }
        }
      } else {
        const int e0 = M.rp[I.row0] + (I.kind == kSegKind ? I.len : 0);
        const int e1 = I.kind == kSegKind ? e0 + I.nrows : I.kind == kOwnKind ? e0 : M.rp[I.row0 + I.nrows];
        if (!far) {
#pragma unroll 2
          for (int k = e0 + lane; k < e1; k += 32) {
            sc[k - e0] = M.ci[k];
            sv[k - e0] = M.v[k];
          }
        }
        if (I.kind <= 32 && lane < I.nrows) {
          const int q = (P ? 0 : C.nlp) + I.len + lane, first = M.rp[I.row0 + lane];
          s_lrp[q] = int2{far ? first : I.ent + first - e0, M.rp[I.row0 + lane + 1] - first};
        }
      }
      if (I.kind != kSegKind && lane < I.nrows) {
        const int row = I.row0 + lane, t = I.vec + lane;
        if (P) {
          s_gp[t] = row;
          pc[t] = v.c[row];
          plo[t] = v.l[row];
          pup[t] = v.u[row];
          pT[t] = v.T[row];
          piT[t] = v.invT[row];
          px[cur * pl.rp + t] = v.x[cur][row];
          if (prm.mode == kPdlp) pxb[t] = v.xbar[cur][row];
        } else {
          s_gd[t] = row;
          db[t] = v.b[row];
          dS[t] = v.S[row];
          diS[t] = v.invS[row];
          dy_[cur * pl.rd + t] = v.y[cur][row];
          dax[cur * pl.rd + t] = v.ax[cur][row];
          if (prm.mode == kPdlp) dyb[t] = v.ybar[cur][row];
          s_sense[t] = d.sense[row];
        }
      }
    }
  }
  if (!kSolo) {
    // Start: every CTA is there, or none does anything.  A CTA that gives up
    // and one that saw the full count agree through one word.
    __syncthreads();
    if (tid == 0) {
      bar_arrive(pl.bar);
      const bool all = bar_wait(pl.bar, arrived + pl.G + missing_arrivals(pl), start_spins(pl));
      const unsigned int was = atomicCAS(pl.bar + 2, 0u, all ? 1u : 2u);
      s_ok = was == 0u ? all : was == 1u;
      if (!s_ok) d.st->fault = 2;
    }
    __syncthreads();
    if (!s_ok) return;
    const int cur = s_st.cur;
    if (kWords)
      for (int t = tid; t < C.rd; t += kResThreads) Elt::put(gyw + (size_t)cur * d.m + s_gd[t], dy_[cur * pl.rd + t], base + 1);
  }
  __syncthreads();

  // One side's row sums, by warps w0, w0 + 1, ...: into sum[local row].
  auto row_sums = [&](const ResItem* it, int n, const V* sv, const int* sc, const int2* lrp, const uint8_t* lens,
                      const CsrT<V>* far, const ResGather<V, kKind>& g, V* sum, int w0) {
    bool ok = true;
#pragma unroll 1
    for (int i = warp - w0; i < n; i += kResWarps - w0) {
      const ResItem& I = it[i];
      if (!kSolo && I.kind == kOwnKind) {  // the segments' sums, in segment order over the lanes
        double t;
        ok = rec_sum(pl.seg + I.ent, I.len, g.seq, g.spins, &t) && ok;
        if (lane == 0) sum[I.vec] = (V)t;
        continue;
      }
      int off, count, most, step = 32;
      if (I.kind == 0) {
        off = I.ent + lane;
        count = lane < I.nrows ? lens[I.vec + lane] : 0;
        most = I.len;
      } else if (!kSolo && I.kind == kSegKind) {
        off = I.ent + lane;
        count = (I.nrows - lane + 31) >> 5;
        most = (I.nrows + 31) >> 5;
      } else {
        const int lg = 31 - __clz(I.kind);
        step = I.kind;
        const int l = lane & (step - 1), r = lane >> lg;
        const bool has = r < I.nrows;
        const int2 e = lrp[I.len + (has ? r : 0)];
        off = e.x + l;
        count = has ? (max(e.y - l, 0) + step - 1) >> lg : 0;
        most = __reduce_max_sync(0xffffffffu, count);
      }
      if constexpr (kSolo && sizeof(V) == 4) {
        if (most > kBlockRowThreshold / 32) {  // (kind 32; a slice's or narrower group's lanes have fewer entries)
          const double w = lane_sum(res_dot_pieces<kKind>(sv + off, sc + off, count, most, g));
          if (lane == 0) sum[I.vec] = (V)w;
          continue;
        }
      }
      V s;
      if (kBars && far) s = res_dot(far->v + off, far->ci + off, count, most, step, g, &ok);
      else s = res_dot(sv + off, sc + off, count, most, step, g, &ok);
      if (I.kind == 0) {
        if (lane < I.nrows) sum[I.vec + lane] = s;
      } else if (!kSolo && I.kind == kSegKind) {
        const double w = lane_sum((double)s);
        if (lane == 0) ResElt<double>::put(pl.seg + I.vec, w, g.seq);
      } else {
        const int lg = 31 - __clz(step);
#pragma unroll 1
        for (int o = step / 2; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o, step);
        if ((lane & (step - 1)) == 0 && (lane >> lg) < I.nrows) sum[I.vec + (lane >> lg)] = s;
      }
    }
    if (!kSolo && !ok) s_ok = 0;
  };
  const CsrT<V> far_a = csr_a<V>(d), far_at = csr_at<V>(d);
  const int wp = min(kResWarps, (C.rp + 31) / 32), wd = min(kResWarps, (C.rd + 31) / 32);  // warps with rows

  unsigned int target = arrived + pl.G;  // arrivals of all CTAs so far
  bool avg = false;  // the last attempt was accepted: its term of the averages is still to be added
  V avg_eta = V(0);
#pragma unroll 1
  for (int a = -1; a < attempts; ++a) {  // (round -1 only forms A^T y)
    const StepScalars<V> sp = read_scalars<V>(&s_st, true);
    const int cur = sp.cur, nxt = a < 0 ? cur : cur ^ 1;
    const bool collect = sp.collect != 0;
    const unsigned int seq = base + 2 + a;  // of this attempt's words (a = -1: the current y)
    V* const yc = dy_ + cur * pl.rd;
    V* const yn = dy_ + nxt * pl.rd;
    if (a >= 0) {
      if ((a % kFacs) == 0 && tid < kFacs)
        step_factors(d.step_tab, s_st.attempts + 1 + tid, &s_fac[0][tid], &s_fac[1][tid]);
      V* const xc = px + cur * pl.rp;
      V* const xn = px + nxt * pl.rp;
      // ---- rows of A^T: x+ -----------------------------------------------------
      V accp[3] = {V(0), V(0), V(0)};
#pragma unroll 1
      for (int t = tid; t < C.rp; t += kResThreads) {
        const int row = s_gp[t];
        if (sp.pend) {  // rare: once every phi accepted steps
          ogd_entry<V>(pT + t, piT + t, v.GT + row, sp.up_scale * v.q[row], prm.sched, (V)prm.alpha, (V)prm.floor,
                       sp.sqrt_gnorm);
          v.T[row] = pT[t];
          v.invT[row] = piT[t];
        }
        const V x0 = xc[t];
        const V g = pc[t] - psum[cur * pl.rp + t];
        const V xh = x0 - sp.step * pT[t] * g;
        const V lo = plo[t], hi = pup[t];
        const auto kx = ord_key(xh), kl = ord_key(lo), kh = ord_key(hi);
        const V x1 = clamp_keys(xh, kx, lo, kl, hi, kh);
        xn[t] = x1;
        if (kWords) Elt::put(gxw + row, x1, seq);
        if (kBars) v.x[nxt][row] = x1;
        const V dx = x1 - x0;
        accp[0] += dx * dx * piT[t];
        if (collect) {
          const V gi = (kx >= kl && kx <= kh) ? g : V(0);
          const V qj = gi * g;
          v.q[row] = qj;
          accp[1] += g * g;
          accp[2] += qj * qj;
        }
      }
      s_red[tid] = (double)accp[0];
      if (!kWords) __syncthreads();
      if (kBars) {
        target += pl.G;
        if (tid == 0) {
          bar_arrive(pl.bar);
          if (!bar_wait(pl.bar, target + missing_words(pl), wait_spins(pl))) s_ok = 0;
        }
        __syncthreads();
        if (!s_ok) {
          if (tid == 0) d.st->fault = 1;
          return;
        }
      }
      // ---- rows of A: A x+ and y+ ------------------------------------------------
      const StepScalars<V> sd = read_scalars<V>(&s_st, false);
      V* const axc = dax + cur * pl.rd;
      V* const axn = dax + nxt * pl.rd;
      row_sums(s_it + np, nd, s_vd, s_cd, s_lrp + C.nlp, s_lend, pl.far & 2 ? &far_a : nullptr,
               ResGather<V, kKind>{kSolo ? xn : v.x[nxt], gxw, seq + missing_words(pl), d.n, d.bad_gathers, wait_spins(pl)}, axn, 0);
      __syncthreads();
      V accd[4] = {V(0), V(0), V(0), V(0)};
#pragma unroll 1
      for (int t = tid; t < C.rd; t += kResThreads) {
        const int row = s_gd[t];
        if (sd.pend) {
          ogd_entry<V>(dS + t, diS + t, v.GS + row, sd.up_scale * v.p[row], prm.sched, (V)prm.alpha, (V)prm.floor,
                       sd.sqrt_gnorm);
          v.S[row] = dS[t];
          v.invS[row] = diS[t];
        }
        const V a1 = axn[t];
        const V a0 = axc[t], bi = db[t], y0 = yc[t];
        const V r = bi - (V(2) * a1 - a0);
        const V yh = y0 + sd.step * dS[t] * r;
        const uint8_t sn = s_sense[t];
        const auto ky = ord_key(yh);
        const bool outside = (sn == kLe && ky > 0) || (sn == kGe && ky < 0);
        const V y1 = outside ? V(0) : yh;
        yn[t] = y1;
        if (kWords) Elt::put(gyw + (size_t)nxt * d.m + row, y1, seq);
        if (kBars) v.y[nxt][row] = y1;
        const V dy = y1 - y0;
        accd[0] += dy * dy * diS[t];
        accd[1] += dy * (a1 - a0);
        if (collect) {
          const V res = bi - a0;
          const V pi = outside ? V(0) : res * r;
          v.p[row] = pi;
          accd[2] += res * res;
          accd[3] += pi * pi;
        }
      }
      // ---- sums ------------------------------------------------------------------
      // fields: dy^2/Sigma, dy.Adx, dx^2/T; then, on attempts that
      // record q and p only (they are 0 otherwise), ||b - A x||^2, sum p^2, ||g||^2, sum q^2
      s_red[kResThreads + tid] = (double)accd[0];
      s_red[2 * kResThreads + tid] = (double)accd[1];
      __syncthreads();
      if (warp < kCtlWarps) {
        const double t = res_sum(s_red + (warp < 2 ? (warp + 1) * kResThreads : 0), warp < 2 ? wd : wp);
        if (lane == 0) s_tot[warp] = t;
      }
      if (collect) {
        __syncthreads();
        s_red[tid] = (double)accd[2];
        s_red[kResThreads + tid] = (double)accd[3];
        s_red[2 * kResThreads + tid] = (double)accp[1];
        s_red[3 * kResThreads + tid] = (double)accp[2];
        __syncthreads();
        if (warp < 4) {
          const double t = res_sum(s_red + warp * kResThreads, warp < 2 ? wd : wp);
          if (lane == 0) s_tot[3 + warp] = t;
        }
        __syncthreads();
      }
    }
    if (warp < kCtlWarps) {
      // ---- totals and step control -------------------------------------------------
      if (a >= 0) {
        bool ok = true;
        __syncwarp();
        if (!kSolo) {
          // field f by warp f % 3: its record out; CTA 0 takes everyone's in
#pragma unroll 1
          for (int f = warp; f < (collect ? 7 : 3); f += kCtlWarps) {
            if (lane == 0) ResElt<double>::put(pl.rec + f * pl.G + blockIdx.x, s_tot[f], seq);
            if (blockIdx.x == 0) {
              __syncwarp();
              double t;
              ok = rec_sum(pl.rec + f * pl.G, pl.G, seq, wait_spins(pl), &t) && ok;
              if (lane == 0) s_tot[f] = t;
            }
          }
          if (!ok) s_ok = 0;
        }
        if (kSolo || blockIdx.x == 0) {
          control_sync();
          if (warp == 0 && (kSolo || s_ok)) {
            if (lane == 0) {
              const double t1[3] = {s_tot[2], collect ? s_tot[5] : 0.0, collect ? s_tot[6] : 0.0};
              const double t2[4] = {s_tot[0], s_tot[1], collect ? s_tot[3] : 0.0, collect ? s_tot[4] : 0.0};
              step_control_state(s_st, prm, s_fac[0][a % kFacs], s_fac[1][a % kFacs], t1, t2);
            }
            if (!kSolo) {  // what the other CTAs' rows read, to every eighth of them
              __syncwarp();
              const double w = bcast_word(s_st, lane & 7);
#pragma unroll 1
              for (int g = lane >> 3; 8 * g < pl.G; g += 4) ResElt<double>::put(pl.ctl + 8 * g + (lane & 7), w, seq);
            }
          }
        } else if (warp == 0) {
          double w = 0.0;
          bool here = false;
          for (int k = 0; k < wait_spins(pl) && !here; ++k)
            here = __all_sync(0xffffffffu, lane >= 8 || ResElt<double>::get(pl.ctl + (blockIdx.x & ~7u) + lane, seq, &w));
          if (!here) s_ok = 0;
          if (lane < 8) bcast_read(s_st, lane, w);
        }
      }
    } else {
      // ---- A^T y+ (or, before the first attempt, A^T y) ----------------------------
      if (kBars && a >= 0) {
        if (tid == 32 * kCtlWarps) {
          bar_arrive(pl.bar);
          if (!bar_wait(pl.bar, target + pl.G, wait_spins(pl))) s_ok = 0;
        }
        rows_sync();
      }
      row_sums(s_it, np, s_vp, s_cp, s_lrp, s_lenp, pl.far & 1 ? &far_at : nullptr,
               ResGather<V, kKind>{kSolo ? yn : v.y[nxt], gyw + (size_t)nxt * d.m, seq, d.m, d.bad_gathers, wait_spins(pl)}, psum + nxt * pl.rp,
               kCtlWarps);
      if (avg) {  // the last accepted attempt's terms of the averages
        const int t0 = tid - 32 * kCtlWarps, step = kResThreads - 32 * kCtlWarps;
#pragma unroll 1
        for (int t = t0; t < C.rp; t += step) pxb[t] = pxb[t] + avg_eta * px[cur * pl.rp + t];
#pragma unroll 1
        for (int t = t0; t < C.rd; t += step) dyb[t] = dyb[t] + avg_eta * yc[t];
      }
    }
    __syncthreads();
    if (!kSolo && !s_ok) {
      if (tid == 0) d.st->fault = 1;
      return;
    }
    if (kBars && a >= 0) target += pl.G;
    avg_eta = sp.eta;
    if (a >= 0) avg = prm.mode == kPdlp && s_st.last_accept != 0;
  }

  // ---- write back -----------------------------------------------------------------
  const int cur = s_st.cur;
#pragma unroll 1
  for (int t = tid; t < C.rp; t += kResThreads) {
    const int row = s_gp[t];
    const V x = px[cur * pl.rp + t];
    v.x[cur][row] = x;
    if (prm.mode == kPdlp) v.xbar[cur][row] = avg ? pxb[t] + avg_eta * x : pxb[t];
  }
#pragma unroll 1
  for (int t = tid; t < C.rd; t += kResThreads) {
    const int row = s_gd[t];
    const V y = dy_[cur * pl.rd + t];
    v.y[cur][row] = y;
    v.ax[cur][row] = dax[cur * pl.rd + t];
    if (prm.mode == kPdlp) v.ybar[cur][row] = avg ? dyb[t] + avg_eta * y : dyb[t];
  }
  if (blockIdx.x == 0) {
    const double* src = reinterpret_cast<const double*>(&s_st);
    double* dst = reinterpret_cast<double*>(d.st);
    constexpr int kFault = (int)(offsetof(DevState, fault) / 8);  // stays as it is: any CTA may have set it
    for (int t = tid; t < (int)(sizeof(DevState) / 8); t += kResThreads)
      if (t != kFault) dst[t] = src[t];
    if (!kSolo && tid == 0) {  // every CTA has read these words and decided (this one has had their records)
      pl.bar[1] = base + 2 + attempts;
      pl.bar[2] = 0u;
      pl.bar[3] = target;
    }
  }
}

template <class V>
const void* resident_fn_t(int kind) {
  if (kind == kSoloKind) return (const void*)resident_kernel<V, kSoloKind>;
  return kind == kWordsKind ? (const void*)resident_kernel<V, kWordsKind> : (const void*)resident_kernel<V, kBarriersKind>;
}
const void* resident_fn(bool fp32, int kind) {
  return fp32 ? resident_fn_t<float>(kind) : resident_fn_t<double>(kind);
}

// Words by default.  A word that many rows gather is one L2 line read that
// often per attempt, where the L1 would serve the plain loads between grid
// barriers: with a column or row of more than kWordsMaxRow entries, barriers
// (the 376k-nonzero LP with rows of up to 3,000 entries: 1,660 us with words,
// 1,112 with barriers; the other way the 60k-nonzero LP, rows of up to 35
// entries: 709 us with words, 779 with barriers, the transportation LP 1,293
// against 1,348).  The line could lie higher for LPs with few long rows: 60k and
// 300k nonzeros with one row in 200 of 140 / 200 / 400 entries, 657 / 670 / 700 and
// 772 / 802 / 822 us with words, 723 / 732 / 748 and 844 / 843 / 870 with barriers
// (the step kernels: 1,290 and 1,470).
constexpr int kWordsMaxRow = 128;
int resident_kind(const ResPlan& pl) {
  if (pl.G == 1) return kSoloKind;
  return pl.longest <= kWordsMaxRow && !pl.far ? kWordsKind : kBarriersKind;
}

}  // namespace

// A resident launch loads its rows, forms A^T y once more and writes its rows back,
// which an attempt or two do not make up for.  us per lp_solve call of one attempt,
// with the step kernels / resident / stepped: 60k nonzeros 78 / 69 / 65,
// transportation 92 / 88 / 83, power law 1M (both matrix copies from L2) 114 / 126 /
// 116; but linking rows 86 / 79 / 81 and power law 100k 83 / 79 / 80.
bool single_attempt_stepped(const ResPlan& pl) { return pl.G > 1 && (resident_kind(pl) == kWordsKind || pl.far == 3); }

// Shortest check period that resident periods are for.  us per attempt with its
// checks, step kernels / resident (one attempt a period: stepped where that is
// the rule above): 1M nonzeros, both copies from L2, a check after every attempt
// 126 / 136, after every second 84 / 87, every fourth 61 / 58; one CTA, every
// attempt 64 / 67, every second 41 / 36; others, every attempt: 60k nonzeros 74 / 66,
// linking rows 88 / 83, transportation 100 / 88, power law 100k 81 / 81.
int shortest_period(const ResPlan& pl) { return pl.far == 3 ? 4 : pl.G == 1 ? 2 : 1; }

// Dynamic shared memory that a resident CTA may take; also lets the stepped kernels have theirs.
cudaError_t resident_smem_limit(int device, int* bytes) {
  int optin = 0;
  cudaError_t e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, device);
  if (e != cudaSuccess) return e;
  int least = optin;
  for (int k = 0; k < 6; ++k) {
    const void* fn = resident_fn(k & 1, k >> 1);
    cudaFuncAttributes at;
    e = cudaFuncGetAttributes(&at, fn);
    if (e != cudaSuccess) return e;
    const int room = optin - (int)at.sharedSizeBytes;
    e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, room);
    if (e != cudaSuccess) return e;
    least = std::min(least, room);
  }
  e = stepped_smem_limit();
  if (e != cudaSuccess) return e;
  *bytes = least;
  return cudaSuccess;
}

cudaError_t launch_resident(const Dev& d, const Params& prm, const ResPlan& pl, bool fp32, int attempts,
                            cudaStream_t s) {
#ifdef LPOP_CHECK_BOUNDS
  if (pl.test.refuse) return cudaErrorCooperativeLaunchTooLarge;
#endif
  Dev da = d;
  Params pa = prm;
  ResPlan pp = pl;
  void* args[] = {&da, &pa, &pp, &attempts};
  const void* fn = resident_fn(fp32, resident_kind(pl));
  if (pl.G == 1) return cudaLaunchKernel(fn, dim3(1), dim3(kResThreads), args, (size_t)pl.smem, s);
  return cudaLaunchCooperativeKernel(fn, dim3((unsigned)pl.G), dim3(kResThreads), args, (size_t)pl.smem, s);
}

SmTokens& sm_tokens(int device, int sms) {
  static std::mutex mu;
  static std::unique_ptr<SmTokens> tokens[64];
  std::lock_guard<std::mutex> lk(mu);
  std::unique_ptr<SmTokens>& t = tokens[device & 63];
  if (!t) t = std::make_unique<SmTokens>(sms);
  return *t;
}

}  // namespace lpop
